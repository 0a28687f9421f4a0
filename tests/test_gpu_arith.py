"""The kernels' own arithmetic, probed on the GPU (tests/cuda/arith.cu, compiled
here from the kernels' headers).

Mixed cell inversion: wherever the float-float form is taken, the cache's T, P,
rho, Y and u are the FP64 form's, bit for bit, over pure, mixed and trace
compositions (down to 1e-14 and, for partial densities below float-float's
range, 1e-30), 3e3 to 3e7 Pa, 200 to 1700 K, from rest to flow whose kinetic
energy is 1000 times its thermal energy, for one liquid, two liquids and a NASG
liquid with covolume and reference energy.  Refusals are legitimate and are
bounded: at low speed, with no species below the range, at most 5 %.

Reciprocals, roots and quotients against CUDA's, over 2^-1000 .. 2^1000 and
mantissas at the ends of the binade: drcp leaves 2^-57 of its series and one
rounding (at most 1 ulp from the rounded quotient), drsqrt the roundings of its
residual and of its last step, 2^-53 (1 + 1/2) (at most 200 of 2^-60), qdiv two
roundings and drcp's (at most 2 ulp), ddiv the division's own result."""
import ctypes
import os
import subprocess

import pytest
import torch

from paper_2504_14063_gb300 import workloads as W

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2504_14063_gb300 import build
    so = str(tmp_path_factory.mktemp("probe") / "arith.so")
    flags = [f for f in build.NVCC_FLAGS if f != "-lineinfo"]
    subprocess.check_call([build._nvcc()] + flags + ["-shared", "-I", build.CSRC, "-I", build.INCLUDE, "-o", so,
                                                     os.path.join(ROOT, "tests", "cuda", "arith.cu")])
    return ctypes.CDLL(so)


def _states(species, D, n, speed, trace):
    """Conserved states [ns + D + 1, n]: kinetic over thermal energy up to `speed`,
    half of the volume fractions traces of 10^-trace .. 1, some species absent."""
    g = torch.Generator("cuda").manual_seed(3)
    r = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)
    ns = len(species)
    w = r(ns, n)
    w = torch.where(r(ns, n) < 0.5, 10.0 ** (-trace * r(ns, n)), w)
    w[torch.randint(ns, (n,), generator=g, device="cuda"), torch.arange(n, device="cuda")] = 1.0
    w = torch.where(r(ns, n) < 0.15, torch.zeros_like(w), w)
    w[0] = torch.where(w.sum(0) == 0, torch.ones_like(w[0]), w[0])
    al = w / w.sum(0)
    P, T = 10.0 ** (3.5 + 4 * r(n)), 200.0 + 1500 * r(n)
    ry = [al[k] / ((s.gamma - 1) * s.cv * T / (P + s.pinf) + s.b) for k, s in enumerate(species)]
    rho = sum(ry)
    th = [s.cv * T * (P + s.gamma * s.pinf) / (P + s.pinf) for s in species]
    et = sum(a * b for a, b in zip(ry, th)) / rho
    u = torch.randn(D, n, generator=g, device="cuda", dtype=torch.float64)
    u = u / u.norm(dim=0) * torch.sqrt(2 * et * speed * r(n))
    E = sum(a * (b + s.q) for a, b, s in zip(ry, th, species)) + 0.5 * rho * (u * u).sum(0)
    return torch.stack(ry + list(rho * u) + [E]).contiguous()


SETS = {"nasg": ([W.WATER_NASG, W.AIR_TABLE], 1), "one_liquid": ([W.AIR, W.HELIUM, W.LIQUID_SG], 2),
        "two_liquids": ([W.LIQUID_SG, W.LIQUID_B, W.AIR, W.HELIUM], 3)}


@pytest.mark.parametrize("name", SETS)
@pytest.mark.parametrize("speed,trace", [(0.01, 14), (1, 14), (30, 14), (1000, 14), (0.01, 30)])
def test_mixed_inversion_is_fp64_rounded(probe, name, speed, trace):
    from paper_2504_14063_gb300 import binding as mp
    species, D = SETS[name]
    U = _states(species, D, 2_000_000, speed, trace)
    per = (W.BC_PERIODIC,) * 3
    p = W.Problem(name, D, tuple([8] * D + [1] * (3 - D)), 1.0, species, W.Model(cdi=1), None, bc_lo=per, bc_hi=per)
    g, e, m = mp.structs_from_problem(p, mp.MIXED)
    out = torch.zeros(8, dtype=torch.int64, device="cuda")
    assert probe.probe_cells(ctypes.byref(g), ctypes.byref(e), ctypes.byref(m), ctypes.c_void_p(U.data_ptr()),
                             ctypes.c_longlong(U.shape[1]), ctypes.c_void_p(out.data_ptr())) == 0
    taken, *differ = out.cpu().tolist()[:7]
    print(f"{name} speed {speed} trace 1e-{trace}: taken {taken / U.shape[1]:.4f}, differing {differ}")
    assert differ == [0] * 6
    if speed <= 1 and trace <= 14:
        assert taken >= 0.95 * U.shape[1]


@pytest.mark.parametrize("kind", ["random", "ends", "near"])
def test_reciprocals_roots_and_quotients(probe, kind):
    n = 8_000_000
    g = torch.Generator("cuda").manual_seed(5)
    r = lambda: torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    if kind == "near":      # ordinary sizes, quotients near one
        b = 1.0 + r()
        a = b * (1.0 + 1e-9 * (r() - 0.5))
    else:
        m = 1.0 + r()
        if kind == "ends":  # within 64 ulp of a power of two, on either side
            m = 1.0 + torch.randint(-64, 65, (n,), generator=g, device="cuda").double() * 2.0 ** -53
        pow2 = lambda lim: ((torch.randint(-lim, lim, (n,), generator=g, device="cuda") + 1023) << 52).view(torch.float64)
        b = m * pow2(999)
        a = (1.0 + r()) * pow2(20)
        b = torch.where(r() < 0.5, -b, b)
    out = torch.zeros(8, dtype=torch.int64, device="cuda")
    assert probe.probe_div(ctypes.c_void_p(a.data_ptr()), ctypes.c_void_p(b.data_ptr()), ctypes.c_longlong(n),
                           ctypes.c_void_p(out.data_ptr())) == 0
    rcp, quo, root, d1, d2 = out.cpu().tolist()[:5]
    print(f"{kind}: drcp {rcp} ulp, qdiv {quo} ulp, drsqrt {root} of 2^-60, ddiv differs {d1} and {d2}")
    assert rcp <= 1 and quo <= 2 and root <= 200 and d1 == 0 and d2 == 0
