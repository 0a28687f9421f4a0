"""Device memory of the reverse passes: what they can do without is allocated
only by the call that uses it and never in the place of what they need."""
import pytest
import torch

from paper_2504_14063_gb300 import workloads as W

pytestmark = pytest.mark.gpu
MB2 = 2 << 20   # the driver's allocation granularity


@pytest.fixture(scope="module")
def mods():
    from paper_2504_14063_gb300 import autograd, binding
    return autograd, binding


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_second_cache_comes_last_and_only_where_it_is_used(mods):
    _, mp = mods
    p = W.random_smooth_2d(nx=640, ny=640, seed=3)
    ctx = mp.Context(p)
    U0 = ctx.init_state(torch.from_numpy(p.prim))
    lam = torch.randn(U0.shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(0))
    dt = 0.5 * float(ctx.dt_gamma(U0)[0])
    tape = torch.empty(3 * ctx.nfaces_total, dtype=torch.int32, device="cuda")
    caches = torch.empty(3 * ctx.cache_doubles, dtype=torch.float64, device="cuda")
    stages = ctx.rk_step_record(U0.clone(), dt, tape, None, caches)
    out, ref, lamW = torch.empty_like(U0), torch.zeros_like(U0), torch.zeros_like(ctx.primitives(U0))
    cache = 8 * ctx.cache_doubles
    assert cache > 16 * MB2
    a = _free()
    ctx.rhs_adjoint(U0, None, None, lam, out)
    b = _free()
    ctx.primitives_adjoint(U0, lamW, out)
    ctx.rk_step_adjoint(U0, lam, dt, tape, out, stages, caches)
    assert _free() == b        # neither takes the cache that it has no use for
    ctx.rk_step_adjoint(U0, lam, dt, tape, ref, stages)
    c = _free()
    assert cache <= b - c <= cache + MB2
    need = a - b               # what the reverse step cannot do without
    # a context with room for that and half a cache
    tight = mp.Context(p)
    left = need + cache // 2
    fill = torch.empty(_free() - left, dtype=torch.uint8, device="cuda")
    try:
        assert need < _free() < need + cache
        tight.rk_step_adjoint(U0, lam, dt, tape, out, stages)
        torch.cuda.synchronize()
    finally:
        del fill
        torch.cuda.empty_cache()
    assert torch.equal(out, ref)
    # (and the attempt is not repeated once there is room)
    d = _free()
    tight.rk_step_adjoint(U0, lam, dt, tape, out, stages)
    assert _free() == d and torch.equal(out, ref)


@pytest.mark.parametrize("n,every", [(12, 4), (10, 4), (9, 9)])
@pytest.mark.parametrize("kept", [False, True])
def test_backward_of_a_rollout_holds_one_segment(mods, monkeypatch, n, every, kept):
    """The backward pass allocates no more than one segment's buffers, kept or
    not, whole or with a shorter last one (measured in torch's allocator, which
    every buffer of it comes from)."""
    ag, mp = mods
    p = W.shock_bubble_2d(nx=256, ny=128, seed=1)
    ctx = mp.Context(p)
    prim = torch.from_numpy(p.prim).cuda().requires_grad_()
    probe = torch.zeros(p.prim.shape[1:], dtype=torch.float64, device="cuda")
    probe[:, :, 80] = 1.0 / 128
    seg = ag._segment
    if not kept:
        monkeypatch.setattr(ag, "_segment", lambda c, m, like, share=None: None if share is not None else seg(c, m, like))
    state = ctx.nv * ctx.ncells * 8
    one = (3 * every + 1) * state + every * 3 * (ctx.nfaces_total * 4 + ctx.cache_doubles * 8)
    U, J, _ = ag.rollout(ctx, ag.init_state(ctx, prim), n, every=every, probe=probe)
    torch.cuda.synchronize()
    base = torch.cuda.memory_allocated()
    torch.cuda.reset_peak_memory_stats()
    g, = torch.autograd.grad(J, prim)
    assert float(g.abs().max()) > 0
    peak = torch.cuda.max_memory_allocated() - base
    print(f"peak {peak / one:.2f} segments")
    # besides the segment: the adjoint, its copies, the probe's field adjoint
    # and the gradient, a few fields of a cell each
    rest = 12 * state
    assert peak <= (0 if kept and n % every == 0 else one) + rest
    assert rest < 0.5 * one


def test_reverse_step_under_capture_allocates_nothing(mods):
    """A reverse step captured before the second cache exists takes the route
    without it, bit for bit the same."""
    _, mp = mods
    p = W.random_smooth_2d(nx=61, ny=47, seed=3)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx = mp.Context(p, stream=s)
        U0 = ctx.init_state(torch.from_numpy(p.prim))
        lam = torch.randn(U0.shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(0))
        dt = 0.5 * float(ctx.dt_gamma(U0)[0])
        out, ref = torch.empty_like(U0), torch.empty_like(U0)
        ctx.rhs_adjoint(U0, None, None, lam, torch.zeros_like(U0))   # the scratch, without the second cache
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        ctx.rk_step_adjoint(U0, lam, dt, None, out)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        ctx.rk_step_adjoint(U0, lam, dt, None, ref)
    s.synchronize()
    assert float(ref.abs().max()) > 0 and torch.equal(out, ref)
