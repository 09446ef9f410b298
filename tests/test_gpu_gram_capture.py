"""A first call of the NUFFT form of Phi^H Phi inside a stream capture: the
call allocates nothing, so it can be captured, and replays give its result."""
import pytest
import torch

from oracle.nufft import NUFFT
from paper_1406_0359_gb300 import synth
from tests._gpu import TOL, host, need_gpu, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_first_nufft_gram_call_can_be_captured(prec):
    from paper_1406_0359_gb300.binding import Operator

    n, M = 64, 3001
    uv = synth.uv_coverage(M, n, 4)
    op = Operator(torch.as_tensor(uv).cuda(), n, 2, prec)
    x = to_dev(synth.random_image(n, 1), prec)
    out = torch.zeros_like(x)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        op.gram(x, 0, out=out)
    x.copy_(to_dev(synth.random_image(n, 2), prec))
    g.replay()
    torch.cuda.synchronize()
    assert rel(host(out), NUFFT(uv, n).gram_real(synth.random_image(n, 2))) < 2 * TOL[prec]
    op.close()
