"""Device memory of a batch's first solve: the instances' set-up scratch in
flight stays within one instance's (or 256 MiB), however many instances there
are.  In a fresh process, whose library pool holds nothing yet."""
import os
import subprocess
import sys

import pytest

from tests._gpu import need_gpu

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_RUN = r"""
import math, sys, threading
import torch
sys.path.insert(0, sys.argv[1])
from paper_1406_0359_gb300.binding import Operator, batch_solve

count, n, M = 8, 1024, 1 << 24
g = torch.Generator(device="cuda").manual_seed(1)
ops, ys = [], []
for k in range(count):
    uv = math.pi * (2 * torch.rand(M, 2, generator=g, device="cuda", dtype=torch.float64) - 1)
    ops.append(Operator(uv, n, 2, "fp32"))
    del uv
    ys.append(torch.randn(M, generator=g, device="cuda", dtype=torch.complex64))
torch.cuda.synchronize()
torch.cuda.empty_cache()
free0 = torch.cuda.mem_get_info()[0]
owned0 = sum(o.info()["device_bytes"] for o in ops)
low, stop = [free0], [False]

def poll():
    while not stop[0]:
        low[0] = min(low[0], torch.cuda.mem_get_info()[0])

t = threading.Thread(target=poll)
t.start()
batch_solve(ops, ys, [1.0] * count, t_max=1, cg_iters=1, nu=1e-3, gamma=1e-3)
stop[0] = True
t.join()
print(free0 - low[0] - (sum(o.info()["device_bytes"] for o in ops) - owned0))
"""


def test_set_up_scratch_does_not_grow_with_the_batch():
    """An instance's scratch: 16 bytes a point, (2n)^2 reals, twice (2n)^2 complex
    values and a half grid of (4n)(2n): 420 MB.  Work items, pool rounding and
    the batch's tables come on top; two instances' would be above 800 MB."""
    need_gpu()
    r = subprocess.run([sys.executable, "-c", _RUN, ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    over = int(r.stdout.strip().splitlines()[-1])
    n2, M = 2048, 1 << 24
    scratch = 16 * M + n2 * n2 * 4 + 2 * n2 * n2 * 8 + (2 * n2 + 8) * (n2 + 8) * 8
    assert over < 1.75 * scratch
