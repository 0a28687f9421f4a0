"""The forward FP64 face pass that splits a face's fields over warps (small 1D
and 2D grids): both sides of the size where it ends, every interpolation,
species count and boundary, counts around a warp; against the oracle with the
bound of test_gpu_parity."""
import pytest

from paper_2504_14063_gb300 import workloads as W
from tests.test_gpu_parity import rhs_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mp():
    from paper_2504_14063_gb300 import binding
    return binding


@pytest.mark.parametrize("n", [33, 9727, 9728])   # (9727 cells have 9728 faces)
@pytest.mark.parametrize("recon", [W.RECON_WENO5Z, W.RECON_WENO5JS, W.RECON_TENO5, W.RECON_TENO6])
def test_1d(mp, n, recon):
    p = W.interface_advection_1d(n=n, cdi=1)
    p.model.recon = recon
    rhs_parity(mp, p, pre_steps=1)


@pytest.mark.parametrize("nx,ny", [(5, 32), (97, 100), (99, 100)])
@pytest.mark.parametrize("recon", [W.RECON_WENO5Z, W.RECON_TENO6])
@pytest.mark.parametrize("bc", [W.BC_WALL, W.BC_PERIODIC])
def test_2d(mp, nx, ny, recon, bc):
    p = W.random_smooth_2d(nx=nx, ny=ny, seed=nx, bc=bc)
    p.model.recon = recon
    rhs_parity(mp, p, pre_steps=1)


def test_one_species(mp):
    rhs_parity(mp, W.sod(100), pre_steps=2)
