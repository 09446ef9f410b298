"""The NUFFT form's buffer of M sorted visibilities is taken by its first use
and kept: an operator that only ever uses Phi, Phi^H and the convolution form
does not hold it."""
import pytest
import torch

from oracle.nufft import NUFFT
from paper_1406_0359_gb300 import synth
from tests._gpu import TOL, host, measured_problem, need_gpu, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()


@pytest.mark.parametrize("prec,size", [("fp32", 8), ("fp64", 16)])
def test_buffer_comes_with_the_first_nufft_form(prec, size):
    from paper_1406_0359_gb300.binding import Operator

    P = measured_problem(64, 30011, 5)
    n, M = P["n"], P["M"]
    op = Operator(torch.as_tensor(P["uv"]).cuda(), n, 2, prec)
    x, y = to_dev(synth.random_image(n, 1), prec), to_dev(P["y"], prec)
    op.phi_adj(op.phi(x))
    op.gram(x, 1)
    kw = dict(t_max=2, cg_iters=2)
    a = op.solve(y, P["eps"], gram=1, **kw)
    before = op.info()["device_bytes"]
    assert rel(host(op.gram(x, 0)), NUFFT(P["uv"], n).gram_real(host(x))) < 2 * TOL[prec]
    assert op.info()["device_bytes"] - before == M * size
    b = op.solve(y, P["eps"], gram=0, **kw)
    op.gram(x, 0)
    assert op.info()["device_bytes"] - before == M * size
    assert rel(host(b.x), host(a.x)) < 1e-4  # the two forms differ by the NUFFT error of the PSF
    op.close()


def test_solve_in_the_nufft_form_takes_the_buffer():
    from paper_1406_0359_gb300.binding import Operator

    P = measured_problem(64, 3001, 6)
    op = Operator(torch.as_tensor(P["uv"]).cuda(), 64, 2, "fp32")
    assert rel(host(op.solve(to_dev(P["y"], "fp32"), P["eps"], gram=0, t_max=2, cg_iters=2).x),
               host(op.solve(to_dev(P["y"], "fp32"), P["eps"], gram=1, t_max=2, cg_iters=2).x)) < 1e-4
    op.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_ball_partials_come_with_several_blocks(prec):
    """One visibility block adds its norms to accumulators; only several blocks
    keep two partial sums per work item, sized again for every new binning."""
    from paper_1406_0359_gb300.binding import Operator

    P = measured_problem(64, 9001, 7)
    op = Operator(torch.as_tensor(P["uv"]).cuda(), 64, 2, prec)
    y = to_dev(P["y"], prec)
    kw = dict(t_max=3, cg_iters=3)
    one = op.solve(y, P["eps"], **kw)
    before = op.info()["device_bytes"]
    ids = torch.arange(9001, device="cuda", dtype=torch.int32)
    op.set_blocks(ids % 3, 3)
    three = op.info()
    assert three["device_bytes"] - before >= 16 * three["n_items"]
    a = op.solve(y, P["eps"], **kw)
    op.set_blocks(ids % 7, 7)
    b = op.solve(y, P["eps"], **kw)
    op.set_blocks(0 * ids, 1)
    again = op.solve(y, P["eps"], **kw)
    assert rel(host(again.x), host(one.x)) < {"fp32": 1e-5, "fp64": 1e-11}[prec]
    for r in (a, b):
        assert rel(host(r.x), host(one.x)) < 0.1  # the same data within per-block bounds
    op.close()
