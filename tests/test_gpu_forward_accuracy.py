"""The forward float-float kernels are no further from extended precision than
the plain FP64 ones: the error of rhs without flags against that of rhs with
flags (the recording kernels), both against the oracle's right-hand side in long
double, per field as L1 sums over the cells.

Bound: the geometric mean of the ratio over eight states at most 1.1.  (Both
errors are sums of some thousand cells' roundings of the same size; of a few
hundred independent ones, a ratio scatters by 5 %, the mean of eight by 2 %, and
1.1 is five times that.)"""
import os

import numpy as np
import pytest
import torch

from oracle import Oracle
from paper_2504_14063_gb300 import workloads as W

pytestmark = pytest.mark.gpu
RK = (1.0, 0.0, 1.0)


def _problem(name, seed):
    if name == "shock_bubble":
        return W.shock_bubble_2d(nx=96, ny=64, seed=seed)
    if name == "shock_droplet":
        return W.shock_droplet_3d(n=20, seed=seed)
    if name == "droplet_field":
        return W.droplet_field_3d(n=18, ndrops=3, seed=seed, rmin=3.0, rmax=5.0)
    return W.random_smooth_2d(nx=60 + seed, ny=50, seed=seed)


@pytest.mark.parametrize("name", ["shock_bubble", "shock_droplet", "droplet_field", "smooth"])
@pytest.mark.parametrize("recon", [W.RECON_WENO5Z, W.RECON_TENO5])
def test_error_against_extended_precision(name, recon):
    from paper_2504_14063_gb300 import binding as mp
    logs = []
    for seed in range(8):
        p = _problem(name, seed)
        p.model.recon = recon
        ctx = mp.Context(p)
        U = ctx.init_state(torch.from_numpy(p.prim))
        ctx.step_n(U, (0, 3, 10, 30)[seed % 4])
        dt, G = ctx.dt_gamma(U).cpu().tolist()
        stage = dict(U_n=U, rk=RK, dt=dt, Gamma=G)
        fl = torch.empty(ctx.nfaces_total, dtype=torch.int32, device="cuda")
        Uh = U.cpu().numpy()
        hi, lo = Oracle(p, nthreads=os.cpu_count() or 4).stage_ext(Uh, Uh, RK, dt, G)
        err = lambda L: np.abs((L.cpu().numpy() - hi) - lo).sum(axis=(1, 2, 3))
        fast, plain = err(ctx.rhs(U, stage=stage)), err(ctx.rhs(U, stage=stage, flags=fl))
        assert np.all(plain > 0)
        logs.append(np.log(fast / plain))
    r = np.exp(np.mean(logs, axis=0))
    print(f"{name} recon {recon}: error ratio per field {np.array2string(r, precision=2)}")
    assert np.all(r <= 1.1)
