"""The plans of the largest sides: the transforms at n = 2048 in both precisions
and tiles against the oracle, and the large-tile SARA kernels over a table of
instances (512^2: the first analysis level; 1024^2: the synthesis too)."""
import numpy as np
import pytest
import torch

from oracle.nufft import NUFFT
from paper_1406_0359_gb300 import synth
from tests._gpu import TOL, host, need_gpu, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()


@pytest.fixture(scope="module")
def oracle_2048():
    """A Gaussian coverage and, beside it, points on and around the fold v = 0 and v = -pi."""
    n, M = 2048, 3001
    cell = np.pi / n
    edge = [(u * cell, v * cell) for u in (-2048, -1024.5, -3, 0, 0.5, 2047) for v in (-2048, -2047.5, -4, -1, 0, 0.5, 3, 2047)]
    uv = np.concatenate([synth.uv_coverage(M, n, 5), np.array(edge)])
    ref = NUFFT(uv, n)
    x, y = synth.random_image(n, 3), synth.random_vis(len(uv), 4)
    return uv, x, y, ref.phi(x), ref.phi_adj_real(y), ref.gram_real(x)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("tile", [8, 16])
def test_transforms_at_2048_match_oracle(oracle_2048, prec, tile):
    from paper_1406_0359_gb300.binding import Operator

    uv, x, y, phi, adj, gram = oracle_2048
    op = Operator(torch.as_tensor(uv).cuda(), 2048, 1, prec, tile=tile, chunk=0)
    assert rel(host(op.phi(to_dev(x, prec))), phi) < TOL[prec]
    assert rel(host(op.phi_adj(to_dev(y, prec))), adj) < TOL[prec]
    assert rel(host(op.gram(to_dev(x, prec), 0)), gram) < 2 * TOL[prec]
    op.close()


@pytest.mark.parametrize("n,levels,mask", [(512, 2, 0x1FF), (512, 4, 0x1E0), (1024, 1, 0x1FF), (1024, 4, 0x1FF), (1024, 3, 0x102)])
def test_large_tiles_over_a_batch_equal_single_solves(n, levels, mask):
    from paper_1406_0359_gb300.binding import Operator, batch_solve

    inst = []
    for k in range(3):
        M = 20011 + 1000 * k
        op = Operator(torch.as_tensor(synth.uv_coverage(M, n, k)).cuda(), n, levels, "fp32")
        op.set_dictionary(mask)
        y = op.phi(to_dev(synth.sky(n, k), "fp32"))
        inst.append((op, y, 0.03 * float(torch.linalg.vector_norm(y))))
    kw = dict(t_max=3, cg_iters=4, n_reweight=1)
    solo = [op.solve(y, e, **kw) for op, y, e in inst]
    got = batch_solve([i[0] for i in inst], [i[1] for i in inst], [i[2] for i in inst], **kw)
    for a, b in zip(got, solo):
        assert rel(host(a.x), host(b.x)) < 1e-5
        assert a.stats["objective"] == pytest.approx(b.stats["objective"], rel=1e-4)
    for op, _, _ in inst:
        op.close()
