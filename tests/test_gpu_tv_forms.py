"""Both forms of the TV block's dual steps in FP32 -- five a launch on haloed
tiles from 512^2 up, one a launch below -- at step counts around a launch's
share, against the same solve in FP64 (whose steps the oracle tests)."""
import pytest
import torch

from paper_1406_0359_gb300 import synth
from tests._gpu import TOL, host, need_gpu, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()


@pytest.mark.parametrize("n", [16, 256, 512])
@pytest.mark.parametrize("tv_iters", [1, 2, 5, 6, 9, 10, 11, 23])
def test_fp32_steps_match_fp64(n, tv_iters):
    """Two iterations of two CG steps and the three blocks apply about ten
    operators, each within TOL of its FP64 form."""
    from paper_1406_0359_gb300.binding import Operator

    M = 10 * n + 1
    uv = torch.as_tensor(synth.uv_coverage(M, n, 7)).cuda()
    x0 = synth.sky(n, 7, 3, 10)
    got = {}
    for prec in ("fp64", "fp32"):
        op = Operator(uv, n, 1, prec)
        y = op.phi(to_dev(x0, "fp64")) if prec == "fp64" else y.to(torch.complex64)
        eps = 0.05 * float(torch.linalg.vector_norm(y))
        if prec == "fp64":  # nu and a gamma large enough to clip the dual, the same for both
            st = op.solve(y, eps, t_max=1, cg_iters=1).stats
            kw = dict(nu=st["nu"], gamma=20 * st["gamma"], t_max=2, cg_iters=2, n_reweight=1)
        op.set_prior("tv", tv_iters)
        got[prec] = op.solve(y, eps, **kw)
        op.close()
    assert rel(host(got["fp32"].x), host(got["fp64"].x)) < 10 * TOL["fp32"]
    assert got["fp32"].stats["objective"] == pytest.approx(got["fp64"].stats["objective"], rel=1e-4)
