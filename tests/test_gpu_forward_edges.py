"""The forward FP64 passes at the sizes where a launch can go wrong: the
smallest grids (three cells, where the six-cell stencil wraps or mirrors over
the whole domain), counts around a warp and a block, ragged boxes, and
stencils of the general FP64 form, against the oracle with the bound of
test_gpu_parity."""
import pytest

from paper_2504_14063_gb300 import workloads as W
from tests.test_gpu_parity import rhs_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mp():
    from paper_2504_14063_gb300 import binding
    return binding


@pytest.mark.parametrize("n", [3, 31, 32, 33, 127, 128, 129, 257])
@pytest.mark.parametrize("cdi", [0, 1])
def test_1d_sizes(mp, n, cdi):
    rhs_parity(mp, W.interface_advection_1d(n=n, cdi=cdi), pre_steps=1)


@pytest.mark.parametrize("nx,ny", [(3, 3), (3, 41), (65, 3), (33, 31)])
@pytest.mark.parametrize("bc", [W.BC_PERIODIC, W.BC_WALL, W.BC_ZEROGRAD])
def test_2d_sizes_and_boundaries(mp, nx, ny, bc):
    rhs_parity(mp, W.random_smooth_2d(nx=nx, ny=ny, seed=nx + ny, bc=bc), pre_steps=1)


@pytest.mark.parametrize("eps", [1e-40, 1e-6, 1e2])
def test_weno_epsilons(mp, eps):
    p = W.shock_bubble_2d(nx=48, ny=24, seed=1)
    p.model.weno_eps = eps
    rhs_parity(mp, p, pre_steps=2)


def test_without_limiter(mp):
    p = W.random_smooth_2d(nx=29, ny=35, seed=4)
    p.model.pos_limiter = 0
    rhs_parity(mp, p, pre_steps=1)


def test_scaled_units(mp):
    """The same gas flow in units where pressures are 1e-14 of Pa's numbers:
    the float-float parts scale their operands and the result follows."""
    p = W.sod(64)
    rhs_parity(mp, p, pre_steps=3)
    q = W.sod(64)
    q.prim[2] *= 1e-14            # P; T = P W / (rho R) keeps its relation through cv
    q.species[0].cv *= 1e-14
    rhs_parity(mp, q, pre_steps=3)
