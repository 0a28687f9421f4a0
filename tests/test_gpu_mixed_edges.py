"""The mixed-precision passes at the sizes where a launch can go wrong (the
smallest grids, counts around a warp and a block, ragged boxes) and on states
that leave the float-float forms' range (partial densities below FP32's, values
half way between two FP32 numbers), against the oracle with the bound of
test_gpu_mixed."""
import os

import numpy as np
import pytest
import torch

from oracle import Oracle
from paper_2504_14063_gb300 import workloads as W
from tests.test_gpu_parity import _gross

pytestmark = pytest.mark.gpu
NTH = os.cpu_count() or 4


@pytest.fixture(scope="module")
def mp():
    from paper_2504_14063_gb300 import binding
    return binding


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def mixed_parity(mp, p, change=lambda U: U, pre=1):
    o = Oracle(p, nthreads=NTH)
    Un = change(o.run(o.init_state(), pre)[0].copy())
    dt, G, _ = o.dt_gamma(Un)
    rk = (1.0, 0.0, 1.0)
    _, Lo, _, st = o.stage(Un, Un, rk, dt, G)
    assert st == 0
    F, _ = o.face_fluxes(Un, Un, rk, dt, G)
    ctx = mp.Context(p, precision=mp.MIXED)
    d = _cuda(Un)
    Lg = ctx.rhs(d, stage=dict(U_n=d, rk=rk, dt=dt, Gamma=G)).cpu().numpy()
    assert ctx.status() == 0
    rng = np.random.default_rng(1)
    J = Un * (1.0 + 2.0 ** -24 * rng.standard_normal(Un.shape))
    T32 = np.abs(o.stage(J, J, rk, dt, G)[1] - Lo).sum(axis=(1, 2, 3))
    num = np.abs(Lg - Lo).sum(axis=(1, 2, 3))
    bound = 1e-4 * np.abs(Lo).sum(axis=(1, 2, 3)) + 1e-7 * _gross(p, F) + 10.0 * T32
    print(f"err/bound {np.array2string(num / np.maximum(bound, 1e-300), precision=2)}")
    assert np.all(num <= bound)


@pytest.mark.parametrize("n", [3, 33, 127, 257])
def test_1d_sizes(mp, n):
    mixed_parity(mp, W.interface_advection_1d(n=n, cdi=1))


@pytest.mark.parametrize("nx,ny", [(3, 3), (65, 3), (33, 31)])
@pytest.mark.parametrize("bc", [W.BC_PERIODIC, W.BC_WALL, W.BC_ZEROGRAD])
def test_2d_sizes_and_boundaries(mp, nx, ny, bc):
    mixed_parity(mp, W.random_smooth_2d(nx=nx, ny=ny, seed=nx + ny, bc=bc))


def test_two_liquids(mp):
    mixed_parity(mp, W.droplet_field_3d(n=15, ndrops=3, seed=3, rmin=2.0, rmax=4.0))


@pytest.mark.parametrize("tiny", [1e-39, 1e-60, 1e-310])
def test_partial_densities_below_fp32(mp, tiny):
    p = W.random_smooth_2d(nx=29, ny=35, seed=4)

    def change(U):
        U[1, :, ::3, ::2] = tiny
        return U
    mixed_parity(mp, p, change)


def test_ties(mp):
    """Every conserved value half way between two FP32 numbers in a third of
    the cells."""
    p = W.random_smooth_2d(nx=31, ny=33, seed=5)

    def change(U):
        f = U[..., ::3].astype(np.float32)
        U[..., ::3] = 0.5 * (f.astype(np.float64) + np.nextafter(f, np.float32(np.inf)).astype(np.float64))
        return U
    mixed_parity(mp, p, change)
