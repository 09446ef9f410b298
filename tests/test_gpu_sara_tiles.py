"""SARA analysis and synthesis where the large-tile kernels take over (image
sides 512 and 1024 in FP32) and next to that boundary: all filters, a few, one;
levels that mix both tile sizes; images at unaligned addresses."""
import numpy as np
import pytest
import torch

from oracle import sara as osara
from paper_1406_0359_gb300 import synth
from tests._gpu import TOL, host, need_gpu, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()


def make_op(n, levels, prec, mask):
    from paper_1406_0359_gb300.binding import Operator

    op = Operator(torch.as_tensor(synth.uv_coverage(64, n, 1)).cuda(), n, levels, prec)
    op.set_dictionary(mask)
    return op


@pytest.mark.parametrize("prec,n,levels,mask", [
    ("fp32", 1024, 4, 0x1FF), ("fp32", 1024, 1, 0x1FE), ("fp32", 1024, 2, 0x105), ("fp32", 512, 3, 0x1FF),
    ("fp32", 512, 1, 0x0F1), ("fp32", 1024, 3, 0x100), ("fp32", 256, 2, 0x1FF), ("fp64", 512, 2, 0x1FF)])
def test_tile_sizes_match_oracle(prec, n, levels, mask):
    bases = [k for k in range(9) if mask >> k & 1]
    op = make_op(n, levels, prec, mask)
    x = synth.random_image(n, n + mask)
    assert rel(host(op.sara_fwd(to_dev(x, prec))), osara.analysis(x, levels, bases)) < TOL[prec]
    d = np.random.default_rng(mask).standard_normal((len(bases), n, n))
    assert rel(host(op.sara_adj(to_dev(d, prec))), osara.synthesis(d, levels, bases)) < TOL[prec]
    op.close()


def test_unaligned_arrays():
    n, levels = 1024, 2
    op = make_op(n, levels, "fp32", 0x1FF)
    x = synth.random_image(n, 5)
    xs = torch.zeros(n * n + 1, device="cuda")[1:].view(n, n)
    xs.copy_(to_dev(x, "fp32"))
    cs = torch.zeros(9 * n * n + 3, device="cuda")[3:].view(9, n, n)
    op.sara_fwd(xs, out=cs)
    ref = osara.analysis(x, levels)
    assert rel(host(cs), ref) < TOL["fp32"]
    out = torch.zeros(n * n + 2, device="cuda")[2:].view(n, n)
    op.sara_adj(cs, out=out)
    assert rel(host(out), x) < TOL["fp32"]
    op.close()
