"""A batch that is refused leaves every operator as it was: no verdict on one
call's data reaches the next, and a solve in progress on an operator whose
set-up was not reached goes on."""
import pytest
import torch

from paper_1406_0359_gb300 import synth
from tests._gpu import host, need_gpu, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()


def problems(count, n=64, M=3000):
    from paper_1406_0359_gb300.binding import Operator

    out = []
    for k in range(count):
        op = Operator(torch.as_tensor(synth.uv_coverage(M, n, k)).cuda(), n, 2, "fp32")
        y = op.phi(to_dev(synth.sky(n, k), "fp32"))
        noise = to_dev(synth.random_vis(M, k + 9), "fp32") * float(torch.linalg.vector_norm(y)) / M ** 0.5 * 0.02
        out.append((op, (y + noise).contiguous(), 0.03 * float(torch.linalg.vector_norm(y))))
    return out


def nan_in(y):
    bad = y.clone()
    bad[7] = complex(float("nan"), 0.0)
    return bad


@pytest.mark.parametrize("bad", [(0, 1), (0, 2), (1, 2), (0, 1, 2)])
def test_every_operator_solves_good_data_after_several_bad_instances(bad):
    from paper_1406_0359_gb300.binding import PurifyError, batch_solve

    ps = problems(3)
    ops, ys, eps = [list(c) for c in zip(*ps)]
    alone = [op.solve(y, e, t_max=3, cg_iters=3) for op, y, e in ps]
    with pytest.raises(PurifyError) as e:
        batch_solve(ops, [nan_in(y) if k in bad else y for k, y in enumerate(ys)], eps, t_max=3, cg_iters=3)
    assert e.value.code == -1
    for op, y, eps_k, a in zip(ops, ys, eps, alone):
        assert rel(host(op.solve(y, eps_k, t_max=3, cg_iters=3).x), host(a.x)) < 1e-5
        op.close()


@pytest.mark.parametrize("reached", [1, 2])
def test_solve_in_progress_on_an_unreached_operator_goes_on(reached):
    """Instance reached - 1 is refused for its bound; the operators after it
    have a solve begun and part way, which finishes as if undisturbed."""
    from paper_1406_0359_gb300.binding import PurifyError, batch_solve

    ps = problems(3)
    ops, ys, eps = [list(c) for c in zip(*ps)]
    alone = [op.solve(y, e, t_max=4, cg_iters=3) for op, y, e in ps]
    for op, y, e in ps[reached:]:
        op.solve_begin(y, e, t_max=4, cg_iters=3)
        assert not op.solve_step(2)
    with pytest.raises(PurifyError) as err:
        batch_solve(ops, ys, [0.0 if k == reached - 1 else e for k, e in enumerate(eps)], t_max=4, cg_iters=3)
    assert err.value.code == -1
    for (op, y, e), a in list(zip(ps, alone))[reached:]:
        assert op.solve_step(2)
        assert rel(host(op.solve_end().x), host(a.x)) < 1e-5
    for op in ops:
        op.close()
