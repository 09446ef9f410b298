"""Batches whose instances share an image side but not their wavelet levels or
dictionary: every instance's result is its own solve's, in the batched solver
and in the request server's batched iterations."""
import pytest
import torch

from paper_1406_0359_gb300 import synth
from tests._gpu import host, measured_problem, need_gpu, rel, to_dev

pytestmark = pytest.mark.gpu

ALL = 0x1FF
# (image side, M, levels, dictionary) of the instances
MIXES = {
    "levels": [(64, 3000, 4, ALL), (64, 2500, 1, ALL), (64, 3001, 4, ALL), (64, 2000, 2, ALL)],
    "dictionaries": [(64, 3000, 3, ALL), (64, 2500, 3, 1), (64, 3001, 3, 1 << 8), (64, 2000, 3, 0x0F)],
    "both, two sides": [(128, 9000, 2, ALL), (64, 2500, 3, 0x101), (128, 9001, 4, 1 << 4), (64, 2000, 3, ALL)],
    # the fewest levels and filters first, and the most first
    "fewest first": [(64, 3000, 1, 1), (64, 2500, 5, ALL)],
    "most first": [(64, 3000, 5, ALL), (64, 2500, 1, 2)],
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-11)])
@pytest.mark.parametrize("mix", list(MIXES))
def test_mixed_levels_and_dictionaries_equal_their_solo_solves(mix, prec, tol):
    from paper_1406_0359_gb300.binding import Operator, batch_solve

    inst = []
    for k, (n, M, levels, mask) in enumerate(MIXES[mix]):
        P = measured_problem(n, M, 40 + k)
        op = Operator(torch.as_tensor(P["uv"]).cuda(), n, levels, prec)
        op.set_dictionary(mask)
        inst.append((op, to_dev(P["y"], prec), P["eps"]))
    kw = dict(t_max=4, cg_iters=4, n_reweight=1)
    solo = [op.solve(y, e, **kw) for op, y, e in inst]
    res = batch_solve([i[0] for i in inst], [i[1] for i in inst], [i[2] for i in inst], **kw)
    for a, b in zip(res, solo):
        assert rel(host(a.x), host(b.x)) < tol
        assert a.stats["objective"] == pytest.approx(b.stats["objective"], rel=10 * tol)
    for op, _, _ in inst:
        op.close()


def test_server_batches_requests_of_mixed_levels():
    from paper_1406_0359_gb300.binding import Server

    ps = [(measured_problem(64, 3000 + k, 50 + k), levels) for k, levels in enumerate((4, 1, 4, 1))]

    def run(batching):
        srv = Server(int(8e9), 8)
        srv.set_batching(batching)
        ids = [srv.submit(P["uv"], P["y"], 64, lv, P["eps"], t_max=6, cg_iters=4, n_reweight=1) for P, lv in ps]
        for _ in range(100000):
            if srv.step() == (0, 0):
                break
        out = [srv.result(i) for i in ids]
        batched = srv.counts()[0]
        srv.close()
        return out, batched

    (on, nb), (off, ns) = run(True), run(False)
    assert nb > 0 and ns == 0
    for a, b in zip(on, off):
        assert a[1]["iterations"] == b[1]["iterations"] == 12
        assert rel(a[0], b[0]) < 1e-5
