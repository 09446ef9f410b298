"""The TV block's dual steps on haloed tiles: step counts around a launch's
share (odd, even, fewer than a launch), image sides from below one tile to
several, weights, against the oracle's solve."""
import math

import pytest
import torch

from oracle import sdmm as osdmm
from oracle import tv as otv
from tests._gpu import host, measured_problem, need_gpu, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()


@pytest.fixture(scope="module", params=[(16, 300), (32, 700), (128, 6001)])
def problem(request):
    n, M = request.param
    P = measured_problem(n, M, 3)
    nu = 1.0 / math.sqrt(osdmm.operator_norm_sq(P["op"], 30))
    P.update(nu=nu, gamma=20 * otv.tv_default_gamma(P["op"], P["y"], nu))  # large enough to clip the dual
    return P


@pytest.mark.parametrize("tv_iters", [1, 4, 5, 6, 10, 11, 23])
@pytest.mark.parametrize("n_rw", [0, 1])
def test_step_counts_match_oracle(problem, tv_iters, n_rw):
    from paper_1406_0359_gb300.binding import Operator

    P = problem
    x_ref, rounds = otv.tv_solve(P["op"], P["y"], P["eps"], P["gamma"], 3, 6, P["nu"], tv_iters, n_rw)
    op = Operator(torch.as_tensor(P["uv"]).cuda(), P["n"], 1, "fp64")
    op.set_prior("tv", tv_iters)
    res = op.solve(to_dev(P["y"], "fp64"), P["eps"], t_max=3, cg_iters=6, n_reweight=n_rw, gamma=P["gamma"], nu=P["nu"],
                   gram=0)
    assert rel(host(res.x), x_ref) < 1e-9
    assert res.stats["objective"] == pytest.approx(rounds[-1].history[-1]["objective"], rel=1e-9)
    op.close()
