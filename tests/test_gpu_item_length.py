"""The default work-item length: FP64 items are half as long as FP32's below
2^14 points (a warp walks an item alone, and in FP64 the walk is the time), and
the operators agree with the oracle when one tile's items meet at its cells."""
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


@pytest.mark.parametrize("prec,longest", [("fp32", 128), ("fp64", 64)])
@pytest.mark.parametrize("n,M", [(32, 512), (64, 129), (256, 2048)])
def test_items_of_one_tile(prec, longest, n, M):
    from paper_1406_0359_gb300.binding import Operator

    # all points in the 8 x 8 tile at cells (8..15, 8..15)
    cell = 2 * np.pi / (2 * n)
    uv = (8 + 8 * np.random.default_rng(n + M).random((M, 2))) * cell
    op = Operator(torch.as_tensor(uv).cuda(), n, 1, prec)
    assert op.info()["n_items"] == -(-M // longest)
    ref = NUFFT(uv, n)
    x, y = synth.random_image(n, 3), synth.random_vis(M, 4)
    assert rel(host(op.phi(to_dev(x, prec))), ref.phi(x)) < TOL[prec]
    assert rel(host(op.phi_adj(to_dev(y, prec))), ref.phi_adj_real(y)) < TOL[prec]
    assert rel(host(op.gram(to_dev(x, prec), 0)), ref.gram_real(x)) < 2 * TOL[prec]
    op.close()
