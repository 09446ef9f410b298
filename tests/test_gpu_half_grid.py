"""The half-grid NUFFT (visibilities of the upper half kept as mirror images)
and the half-length transforms: every transform plan (image side) and both
tile sizes against the oracle, coverages on the fold, and the checkpoint's z_3
in the whole grid's sorted order."""
import math

import numpy as np
import pytest
import torch

from oracle import sdmm as S
from oracle.nufft import NUFFT
from paper_1406_0359_gb300 import synth
from tests._gpu import TOL, host, measured_problem, need_gpu, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()


def make_op(uv, n, prec, tile=0, chunk=0):
    from paper_1406_0359_gb300.binding import Operator

    return Operator(torch.as_tensor(uv).cuda(), n, 1, prec, tile=tile, chunk=chunk)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("n,M", [(16, 33), (32, 1), (64, 1000), (128, 3001), (256, 9999), (512, 20011), (1024, 30001)])
def test_every_plan_matches_oracle(prec, tile, n, M):
    uv = synth.uv_coverage(M, n, n + M)
    op = make_op(uv, n, prec, tile=tile, chunk=256)
    ref = NUFFT(uv, n)
    x = synth.random_image(n, 3)
    y = synth.random_vis(M, 4)
    assert rel(host(op.phi(to_dev(x, prec))), ref.phi(x)) < TOL[prec]
    assert rel(host(op.phi_adj(to_dev(y, prec))), ref.phi_adj_real(y)) < TOL[prec]
    assert rel(host(op.gram(to_dev(x, prec), 0)), ref.gram_real(x)) < 2 * TOL[prec]
    op.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_points_on_the_fold(prec):
    """Grid nodes and half cells on and beside v = 0 and v = -pi, at every
    row edge: cells whose taps cross the half grid's boundary or its mirror."""
    n = 32
    cell = 2 * math.pi / (2 * n)
    vs = [k * cell for k in (-32, -31.5, -31, -30.5, -4, -3.5, -1, -0.5, 0, 0.5, 1, 3, 4, 30, 31, 31.5)]
    us = [k * cell for k in (-32, -31.25, -4, -1, 0, 0.75, 3, 5, 31, 31.5)]
    uv = np.array([(u, v) for u in us for v in vs])
    ref = NUFFT(uv, n)
    op = make_op(uv, n, prec)
    x = synth.random_image(n, 5)
    y = synth.random_vis(len(uv), 6)
    assert rel(host(op.phi(to_dev(x, prec))), ref.phi(x)) < TOL[prec]
    assert rel(host(op.phi_adj(to_dev(y, prec))), ref.phi_adj_real(y)) < TOL[prec]
    op.close()


def test_unaligned_images_are_accepted():
    """Images at an address that is not a multiple of 16 bytes."""
    n, M = 64, 500
    uv = synth.uv_coverage(M, n, 2)
    op = make_op(uv, n, "fp32")
    ref = NUFFT(uv, n)
    x = synth.random_image(n, 1)
    buf = torch.zeros(n * n + 3, device="cuda")
    xs = buf[3:].view(n, n)
    xs.copy_(to_dev(x, "fp32"))
    assert xs.data_ptr() % 16 == 12
    y = op.phi(xs)
    assert rel(host(y), ref.phi(x)) < TOL["fp32"]
    out = torch.zeros(n * n + 1, device="cuda")[1:].view(n, n)
    assert rel(host(op.phi_adj(y, out=out)), ref.phi_adj_real(host(y))) < TOL["fp32"]
    op.close()


def _whole_grid_order(uv, n, blocks=None, TB=8):
    K = 2 * n
    t = np.floor((uv * float(K)) / (2.0 * math.pi)).astype(np.int64) % K
    tile = (t[:, 0] // TB) * (K // TB) + t[:, 1] // TB
    keys = (np.arange(len(uv)), t[:, 1] % TB, t[:, 0] % TB, tile) + ((blocks,) if blocks is not None else ())
    return np.lexsort(keys)


@pytest.mark.parametrize("R", [1, 3])
def test_checkpoint_keeps_the_whole_grid_order(R):
    """z_3 of a saved state against the oracle's, in the order of a stable sort
    by (block, 8 x 8 tile, cell) over the whole grid; then the same state
    loaded into a fresh solve saves to the same bytes."""
    n, M, iters = 64, 2000, 3
    p = measured_problem(n, M, 7)
    uv, y = p["uv"], p["y"]
    blocks = (np.arange(M) % R).astype(np.int32)
    nu = 1.0 / math.sqrt(S.operator_norm_sq(p["op"], 30))
    psi = S.SaraDictionary(1)
    gamma = S.default_gamma(p["op"], psi, y, nu)
    eps = 0.5 * p["eps"]
    idx = [np.nonzero(blocks == b)[0] for b in range(R)]
    bl = (idx, [eps * math.sqrt(len(i) / M) for i in idx]) if R > 1 else None
    st = S.sdmm_init(p["op"], psi, np.zeros((n, n)), nu)
    w = np.ones_like(st.z1)
    for _ in range(iters):
        S.sdmm_iteration(st, p["op"], psi, y, eps, gamma, w, 10, nu, bl)

    def begun():
        op = make_op(uv, n, "fp64")
        if R > 1:
            op.set_blocks(blocks, R)
        op.solve_begin(to_dev(y, "fp64"), eps, t_max=10, cg_iters=10, gamma=gamma, nu=nu)
        return op

    op = begun()
    op.solve_step(iters)
    state = op.save_state()
    op.close()
    z3 = np.frombuffer(state[-16 * M:], dtype=np.complex128)
    order = _whole_grid_order(uv, n, blocks if R > 1 else None)
    assert rel(z3, st.z3[order]) < 1e-4  # the composite's PSF is 1e-7 from the oracle's NUFFT form
    op = begun()
    op.load_state(state)
    assert op.save_state() == state
    op.close()
