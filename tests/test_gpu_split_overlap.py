"""The split solve directly behind the kernel that writes its source, on one stream and with the source
changing every time: the operators let their successor start early, so a split kernel that took its
source before the wait would see the last call's.  Bitwise against the same calls with the device
idle between them; the velocity refresh on a split plan against its three parts (the two plans may
keep different near-field forms, each within 1e-6 of the exact solve; the curl of the difference of
two potentials of the field's own size at dx = 1 stays below 1e-5)."""
import numpy as np
import pytest

from tests.helpers import built, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOLN = np.array([[x, y, z] for z in range(4) for y in range(5) for x in range(5) if (x + y + z) % 4], dtype=np.int32)
N = 6  # inputs


def _setup(**plan_args):
    lgf = built()
    rk = lgf.RKPlan(16, SOLN, 1.0, 0.01, 100.0, poisson_method=2)
    xs = rk.blocks(0)
    t = lgf.Table(lgf.LAPLACE7, max_offset=31)
    plan = lgf.Plan(t, [lgf.Solve(16, 3, SOLN, xs, dx=1.0, scale=-1.0)], method=1, **plan_args)
    gen = torch.Generator("cuda").manual_seed(3)
    us = [torch.randn((len(xs), 3, 16, 16, 16), device="cuda", generator=gen) for _ in range(N)]
    assert np.array_equal(xs[:len(SOLN)], SOLN)
    return rk, plan, us, t


@pytest.mark.parametrize("near_form,far_precision", [(1, 0), (2, 0), (3, 0), (0, 1)])
def test_solve_behind_curl(near_form, far_precision):
    rk, plan, us, _t = _setup(near_form=near_form, far_precision=far_precision)
    w = torch.empty_like(us[0])

    def run(wait):
        out = []
        for u in us:
            a = torch.empty_like(u)
            rk.op(0, u, w)
            wait()
            plan.execute([w[:len(SOLN)]], [a])
            wait()
            out.append(a)
        torch.cuda.synchronize()
        return out

    idle = run(torch.cuda.synchronize)
    for _ in range(4):
        for a, b in zip(run(lambda: None), idle):
            assert torch.equal(a, b)
    plan.check()


def test_refresh_on_split_plan():
    rk, plan, us, _t = _setup()
    ref = []
    for u in us:
        w, a, v = torch.empty_like(u), torch.empty_like(u), torch.empty_like(u)
        for call in (lambda: rk.op(0, u, w), lambda: plan.execute([w[:len(SOLN)]], [a]), lambda: rk.op(1, a, v)):
            call()
            torch.cuda.synchronize()
        ref.append(v)
    first = None
    for _ in range(4):
        got = [torch.empty_like(u) for u in us]
        for u, v in zip(us, got):
            rk.refresh(u, v)
        torch.cuda.synchronize()
        first = first or got
        for v, f, r in zip(got, first, ref):
            assert torch.equal(v, f)
            assert rel_l2(v.cpu().numpy(), r.cpu().numpy()) < 1e-5
