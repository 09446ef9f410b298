"""The batched solver's set-up, run part by part over its instances: nu and
gamma computed, given, or given for some; a bad instance refused without harm
to the others' operators; CG step counts of either parity."""
import numpy as np
import pytest
import torch

from paper_1406_0359_gb300 import synth
from tests._gpu import host, need_gpu, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    need_gpu()


def problems(sizes):
    from paper_1406_0359_gb300.binding import Operator

    out = []
    for k, (n, M) in enumerate(sizes):
        op = Operator(torch.as_tensor(synth.uv_coverage(M, n, k)).cuda(), n, 2, "fp32")
        y = op.phi(to_dev(synth.sky(n, k), "fp32"))
        noise = to_dev(synth.random_vis(M, k + 9), "fp32") * float(torch.linalg.vector_norm(y)) / M ** 0.5 * 0.02
        out.append((op, (y + noise).contiguous(), 0.03 * float(torch.linalg.vector_norm(y))))
    return out


@pytest.mark.parametrize("cg", [1, 2, 5, 10])
def test_batch_equals_single_solves(cg):
    from paper_1406_0359_gb300.binding import batch_solve

    ps = problems([(64, 3000), (128, 9001), (64, 2500)])
    alone = [op.solve(y, e, t_max=4, cg_iters=cg) for op, y, e in ps]
    for nus, gammas in (([0.0] * 3, [0.0] * 3),
                        ([alone[0].stats["nu"], 0.0, alone[2].stats["nu"]], [0.0, 0.0, alone[2].stats["gamma"]])):
        got = batch_solve([p[0] for p in ps], [p[1] for p in ps], [p[2] for p in ps], t_max=4, cg_iters=cg, nu=nus,
                          gamma=gammas)
        for g, a in zip(got, alone):
            assert g.stats["nu"] == pytest.approx(a.stats["nu"], rel=1e-6)
            assert g.stats["gamma"] == pytest.approx(a.stats["gamma"], rel=1e-5)
            assert rel(host(g.x), host(a.x)) < 1e-5
    for p in ps:
        p[0].close()


def test_bad_instance_is_refused_and_the_rest_stay_usable():
    from paper_1406_0359_gb300.binding import PurifyError, batch_solve

    ps = problems([(64, 3000), (64, 2500)])
    bad = ps[1][1].clone()
    bad[7] = complex(float("nan"), 0.0)
    with pytest.raises(PurifyError) as e:
        batch_solve([p[0] for p in ps], [ps[0][1], bad], [p[2] for p in ps], t_max=3, cg_iters=3)
    assert e.value.code == -1
    got = batch_solve([p[0] for p in ps], [p[1] for p in ps], [p[2] for p in ps], t_max=3, cg_iters=3)
    for g, (op, y, eps) in zip(got, ps):
        assert rel(host(g.x), host(op.solve(y, eps, t_max=3, cg_iters=3).x)) < 1e-5
        op.close()
