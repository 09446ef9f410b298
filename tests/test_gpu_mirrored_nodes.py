"""FP32 positions of exact grid nodes: a node of the upper half is kept as its
mirror image with offset 1."""
import math

import numpy as np
import pytest
import torch

from tests._gpu import host, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()


def test_offset_one_is_kept():
    """A point just below a lower node (offset rounds to 1 in the cell before),
    one a unit of 2^-24 further away, and the node's partner -k: the first two are
    told apart, and the partner is the first's mirror image bit for bit wherever
    its coordinate in radians comes out as the node exactly."""
    from paper_1406_0359_gb300.binding import Operator

    n = 256
    cells = np.random.default_rng(1).integers(1, n, (20000, 2)).astype(float)
    x = torch.zeros(n, n, device="cuda")
    x[n // 2 + 72, n // 2 + 72] = 1.0
    y = []
    for c in (cells - 2.0 ** -30, cells - 0.75 * 2.0 ** -24, -cells):
        op = Operator(torch.as_tensor(c * (math.pi / n)).cuda(), n, 2, "fp32")
        y.append(host(op.phi(x)))
        op.close()
    below, further, partner = y
    assert (below != further).mean() > 0.5
    exact = (-cells * (math.pi / n) * (2.0 * n) / (2.0 * math.pi) == -cells).all(1)
    assert exact.mean() > 0.5 and np.array_equal(partner[exact], below[exact].conj())
