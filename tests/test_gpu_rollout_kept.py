"""The rollout whose forward pass records its last segment for the backward
pass: value, step lengths and gradient are those of the rollout that replays
every segment, bit for bit, for whole, ragged and single segments, fixed and
CFL steps; a second backward pass over the same graph gives the same gradient.
The reverse step gives the same with recorded, recomputed and kept caches."""
import pytest
import torch

from paper_2504_14063_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mods():
    from paper_2504_14063_gb300 import autograd, binding
    return autograd, binding


def _run(ag, ctx, prim, probe, n, every, dt):
    p = prim.clone().requires_grad_()
    U, J, dts = ag.rollout(ctx, ag.init_state(ctx, p), n, every=every, probe=probe, dt=dt)
    g, = torch.autograd.grad(J, p, retain_graph=True)
    g2, = torch.autograd.grad(J, p)
    return U.detach(), J.detach(), dts, g, g2


@pytest.mark.parametrize("n,every", [(1, 4), (4, 2), (5, 2), (3, 7)])
@pytest.mark.parametrize("fixed", [False, True])
def test_kept_segment_is_the_replayed_one(mods, monkeypatch, n, every, fixed):
    ag, mp = mods
    p = W.shock_bubble_2d(nx=48, ny=24, seed=1)
    ctx = mp.Context(p)
    prim = torch.from_numpy(p.prim).cuda()
    probe = torch.zeros(prim.shape[1:], dtype=torch.float64, device="cuda")
    probe[:, :, 16] = 1.0 / 24
    dt = 0.5 * float(ctx.dt_gamma(ctx.init_state(prim))[0]) if fixed else 0.0
    a = _run(ag, ctx, prim, probe, n, every, dt)
    seg = ag._segment
    monkeypatch.setattr(ag, "_segment", lambda c, m, like, share=None: None if share is not None else seg(c, m, like))
    b = _run(ag, ctx, prim, probe, n, every, dt)
    assert float(a[3].abs().max()) > 0
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    assert torch.equal(a[3], a[4]) and torch.equal(b[3], b[4])


def test_reverse_step_with_and_without_what_was_recorded(mods):
    ag, mp = mods
    p = W.random_smooth_2d(nx=35, ny=29, seed=3)
    ctx = mp.Context(p)
    U0 = ctx.init_state(torch.from_numpy(p.prim).cuda())
    U = U0.clone()
    tape = torch.empty(3 * ctx.nfaces_total, dtype=torch.int32, device="cuda")
    caches = torch.empty(3 * ctx.cache_doubles, dtype=torch.float64, device="cuda")
    dt = torch.empty(1, dtype=torch.float64, device="cuda")
    stages = ctx.rk_step_record(U, 0.0, tape, None, caches, dt)
    dt2 = torch.empty_like(dt)
    assert torch.equal(ctx.rk_step_replay(U0.clone(), 0.0, dt2), U) and torch.equal(dt, dt2)
    lam = torch.randn(U.shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(0))
    ref = ctx.rk_step_adjoint(U0, lam, tape=tape, stages=stages, wstages=caches)
    for kw in (dict(tape=tape, stages=stages), dict(stages=stages), dict(tape=tape), dict()):
        assert torch.equal(ctx.rk_step_adjoint(U0, lam, **kw), ref), kw
