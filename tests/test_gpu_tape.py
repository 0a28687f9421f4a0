"""A call's limiter flags belong to the arithmetic that the reverse pass
recomputes in: with a tape, rk_step takes the recorded step bit for bit and its
tape and CFL step serve rk_step_adjoint as the recorded ones do; with flags,
rhs takes the first stage of that step.  Calls without them run the
float-float kernels: their right-hand sides against the oracle, at the sizes,
interpolations and limits that test_gpu_forward_edges takes with flags, with
test_gpu_parity's bound."""
import types

import pytest
import torch

from paper_2504_14063_gb300 import workloads as W
from tests.test_gpu_parity import rhs_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mp():
    from paper_2504_14063_gb300 import binding
    return binding


@pytest.mark.parametrize("recon", [W.RECON_WENO5Z, W.RECON_TENO5])
@pytest.mark.parametrize("dt_scale", [0.0, 0.5, 1.3])   # CFL step; fixed ones
def test_rk_step_with_a_tape_is_the_recorded_step(mp, recon, dt_scale):
    p = W.shock_bubble_2d(nx=96, ny=48, seed=2)
    p.model.recon = recon
    ctx = mp.Context(p)
    U0 = ctx.init_state(torch.from_numpy(p.prim))
    ctx.step_n(U0, 30)
    dt = dt_scale * float(ctx.dt_gamma(U0)[0])
    lam = torch.randn(U0.shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(0))
    t1, t2 = (torch.full((3 * ctx.nfaces_total,), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    a, b = U0.clone(), U0.clone()
    stages = ctx.rk_step_record(a, dt, t1)
    ctx.rk_step(b, dt, t2)
    assert int((t1 != 0).sum()) > 0
    assert torch.equal(a, b) and torch.equal(t1, t2)
    ref = ctx.rk_step_adjoint(U0, lam, dt, t1, stages=stages)
    assert torch.equal(ctx.rk_step_adjoint(U0, lam, dt, t2), ref)
    # the right-hand side with flags: the step's first stage
    fl = torch.full((ctx.nfaces_total,), -1, dtype=torch.int32, device="cuda")
    used = torch.empty(1, dtype=torch.float64, device="cuda")
    assert torch.equal(ctx.rk_step_replay(U0.clone(), dt, used), a)
    L = ctx.rhs(U0, stage=dict(rk=(1.0, 0.0, 1.0), dt=float(used)), flags=fl)
    assert torch.equal(fl, t1[:ctx.nfaces_total])
    s = (L * used + U0 - stages[0]).abs().amax((1, 2, 3)) / stages[0].abs().amax((1, 2, 3)).clamp_min(1e-300)
    assert float(s.max()) <= 8 * 2.0 ** -53     # (the update contracts dt / dx with the flux differences)


def _without_flags(mp):
    """A binding whose right-hand sides are those of the call without flags."""
    class Context(mp.Context):
        def rhs(self, U, dUdt=None, stage=None, flags=None):
            super().rhs(U, None, stage, flags)
            return super().rhs(U, dUdt, stage)
    return types.SimpleNamespace(Context=Context)


@pytest.mark.parametrize("n", [3, 31, 32, 33, 127, 129, 257, 9727, 9728])
@pytest.mark.parametrize("cdi", [0, 1])
def test_1d_sizes(mp, n, cdi):
    rhs_parity(_without_flags(mp), W.interface_advection_1d(n=n, cdi=cdi), pre_steps=1)


@pytest.mark.parametrize("nx,ny", [(3, 3), (3, 41), (65, 3), (33, 31)])
@pytest.mark.parametrize("bc", [W.BC_PERIODIC, W.BC_WALL, W.BC_ZEROGRAD])
def test_2d_sizes_and_boundaries(mp, nx, ny, bc):
    rhs_parity(_without_flags(mp), W.random_smooth_2d(nx=nx, ny=ny, seed=nx + ny, bc=bc), pre_steps=1)


@pytest.mark.parametrize("recon", [W.RECON_WENO5Z, W.RECON_WENO5JS, W.RECON_TENO5, W.RECON_TENO6])
def test_interpolations(mp, recon):
    p = W.shock_bubble_2d(nx=100, ny=52, seed=1)
    p.model.recon = recon
    rhs_parity(_without_flags(mp), p, pre_steps=60)


@pytest.mark.parametrize("eps", [1e-40, 1e-6, 1e2])
def test_weno_epsilons(mp, eps):
    p = W.shock_bubble_2d(nx=48, ny=24, seed=1)
    p.model.weno_eps = eps
    rhs_parity(_without_flags(mp), p, pre_steps=2)


def test_without_limiter(mp):
    p = W.random_smooth_2d(nx=29, ny=35, seed=4)
    p.model.pos_limiter = 0
    rhs_parity(_without_flags(mp), p, pre_steps=1)


def test_scaled_units(mp):
    q = W.sod(64)
    q.prim[2] *= 1e-14            # P; T = P W / (rho R) keeps its relation through cv
    q.species[0].cv *= 1e-14
    rhs_parity(_without_flags(mp), q, pre_steps=3)


def test_viscous_and_diffusive(mp):
    p = W.random_smooth_2d(41, 35, seed=5, cdi=1, diffusion=1)
    p.model.viscous = 1
    p.model.mu_liquid = 1e-1
    for s in p.species:
        s.mu *= 1e3
    rhs_parity(_without_flags(mp), p, pre_steps=2)


@pytest.mark.parametrize("p", [W.droplet_field_3d(n=22, ndrops=4, seed=2, rmin=3.0, rmax=5.0),
                               W.shock_droplet_3d(n=24, seed=4)], ids=lambda p: p.name)
def test_3d(mp, p):
    rhs_parity(_without_flags(mp), p, pre_steps=2)
