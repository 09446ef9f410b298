"""Passes chained by dependent launch are no slower than the same passes one
after the other.

With kernel timing on, events stand between the passes and nothing overlaps;
off, each pass may start early.  The chain saves launch latencies, so its time
stays below the sum of the passes' (a fifth is left for noise); CTAs that start
early on few SMs and leave others idle would show as a chain slower than that
(1.5 times the sum for FP64 at n = 512 when every pass let the next one start)."""
import ctypes

import pytest
import torch

from paper_1406_0359_gb300 import synth
from tests._gpu import need_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()


def chained_us(call, reps=20):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(5):
        torch.cuda.synchronize()
        a.record()
        for _ in range(reps):
            call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / reps * 1e3)
    return best


def summed_us(op, call, reps=20):
    from paper_1406_0359_gb300 import binding

    L = binding.lib()
    best = float("inf")
    for _ in range(3):
        L.purify_profile(op.h, 1)
        for _ in range(reps):
            call()
        torch.cuda.synchronize()
        total = 0.0
        for kind in range(15):
            ms, cnt = ctypes.c_double(), ctypes.c_int64()
            L.purify_profile_read(op.h, kind, ctypes.byref(ms), ctypes.byref(cnt))
            total += ms.value
        L.purify_profile(op.h, 0)
        best = min(best, total / reps * 1e3)
    return best


@pytest.mark.parametrize("prec,n", [("fp32", 512), ("fp64", 256), ("fp64", 512), ("fp64", 1024)])
def test_chain_of_passes_is_no_slower_than_their_sum(prec, n):
    from paper_1406_0359_gb300.binding import Operator

    M = 3000
    op = Operator(torch.as_tensor(synth.uv_coverage(M, n, 3)).cuda(), n, 1, prec)
    x = to_dev(synth.random_image(n, 1), prec)
    out, y = torch.empty_like(x), op.phi(x)
    for call in (lambda: op.gram(x, 1, out=out), lambda: op.phi(x, out=y), lambda: op.phi_adj(y, out=out)):
        call()
        alone = summed_us(op, call)
        assert chained_us(call) < 1.2 * alone
    op.close()
