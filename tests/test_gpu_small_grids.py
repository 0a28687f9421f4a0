"""The forward FP64 face pass that splits a face's fields over warps (small 1D
and 2D grids).  A field that is periodic in y and small enough for it is tiled
to a grid beyond its range: the right-hand side has to be the tiled one bit for
bit (the same functions of the same cells), for every interpolation, at counts
around a warp and both sides of the size where the split ends.  In 1D, where
nothing can be tiled without changing x's boundary, both sides of that size
against the oracle with the bound of test_gpu_parity."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2504_14063_gb300 import workloads as W
from tests.test_gpu_parity import rhs_parity

pytestmark = pytest.mark.gpu
ALL = [W.RECON_WENO5Z, W.RECON_WENO5JS, W.RECON_TENO5, W.RECON_TENO6]


@pytest.fixture(scope="module")
def mp():
    from paper_2504_14063_gb300 import binding
    return binding


@pytest.mark.parametrize("n", [33, 9727, 9728])   # (9727 cells have 9728 faces)
@pytest.mark.parametrize("recon", ALL)
def test_1d(mp, n, recon):
    p = W.interface_advection_1d(n=n, cdi=1)
    p.model.recon = recon
    rhs_parity(mp, p, pre_steps=1)


def _rhs(mp, p, U, dt, G):
    ctx = mp.Context(p)
    d = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    return ctx.rhs(d, stage=dict(U_n=d, rk=(1.0, 0.0, 1.0), dt=dt, Gamma=G)).cpu().numpy()


@pytest.mark.parametrize("nx,ny", [(5, 7), (32, 31), (97, 98), (63, 152)])
@pytest.mark.parametrize("recon", ALL)
@pytest.mark.parametrize("cdi,diffusion,viscous", [(1, 1, 1), (0, 0, 0)])
def test_2d_is_the_whole_face_form(mp, nx, ny, recon, cdi, diffusion, viscous):
    p = W.random_smooth_2d(nx=nx, ny=ny, seed=nx, cdi=cdi, diffusion=diffusion)
    p.model.recon, p.model.viscous = recon, viscous
    ctx = mp.Context(p)
    U = ctx.init_state(torch.from_numpy(p.prim))
    dt, G = ctx.dt_gamma(U).cpu().tolist()
    U = U.cpu().numpy()
    t = 9728 // (nx * ny) + 2      # beyond two blocks per SM
    q = dataclasses.replace(p, n=(nx, ny * t, 1), prim=np.tile(p.prim, (1, 1, t, 1)))
    a, b = _rhs(mp, p, U, dt, G), _rhs(mp, q, np.tile(U, (1, 1, t, 1)), dt, G)
    assert np.isfinite(a).all() and np.abs(a).max() > 0
    assert np.array_equal(np.tile(a, (1, 1, t, 1)), b)
