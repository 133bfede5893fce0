"""Q_v of one column (its own kernel) against the moment fields, and the latest
record with its profile, over storage types, columns, row counts around the
kernel's 256 threads, and the state before and after the first step.

Tolerance of Q_v, derived: a row's u_x = J_x / rho; the moment fields round the
species momenta, their product with the density and the quotient to FP32, at
most eight roundings of 2^-24 of the species velocities; beyond that both sum in
FP64."""
import math
import time

import numpy as np
import pytest

from paper_1603_08221_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [binding.LBM_FP32, binding.LBM_BF16, binding.LBM_FP16])
@pytest.mark.parametrize("N,Nx,periodic", [(2, 6, 0), (16, 100, 0), (257, 40, 0), (33, 64, 1)])
def test_volume_flow_of_every_kind_of_column(storage, N, Nx, periodic):
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.2, Kn_out=0.3,
                         storage=storage, x_periodic=periodic, wall=periodic)
    g = binding.LbmMix(**p)
    g.set_accommodation_field(workloads.random_accommodation(Nx, seed=2, spread=0.2))
    f = workloads.random_post_state(N, Nx, seed=4, lo=0.099, hi=0.101)
    f[:, 0] *= 4.0
    g.set_post_state(f.astype(np.float32))
    for steps in (0, 3):
        g.step(steps)
        m = g.moments()
        for x in (1, Nx // 2, Nx - 2):
            ra, rb, ua, ub = (m[k][:, x] for k in ("rho_a", "rho_b", "ua_x", "ub_x"))
            ref = ((ra * ua + rb * ub) / (ra + rb)).sum()
            tol = 8 * 2.0 ** -24 * (np.abs(ua) + np.abs(ub)).sum()
            assert abs(g.volume_flow(x) - ref) <= tol, (steps, x)
    assert g.volume_flow() == g.volume_flow(0 if periodic else Nx - 2)


def test_latest_record_is_the_last_of_the_history():
    p = workloads.preset("heli_argon_320x16", N=8, N_x=300)
    g = binding.LbmMix(**p)
    g.init()
    for n in (1, 12, 300):
        g.step(n)
        s, rec = g.separation(), g.history(1)[0]
        assert [s["CL"], s["Cl_tilde"], s["mdot_a"], s["mdot_b"], s["x_min"]] == list(rec[1:6])
        prof = s["Cl_profile"]
        assert prof.shape == (300,) and prof[0] == p["C_l"] and prof[-1] == p["C_l"]
        assert s["x_min"] == 1 + np.argmin(prof[1:-1])
        assert s["CL"] == (p["C_l"] - prof[1:-1].min()) / p["C_l"]


# both sides of the line beyond which the profile is a copy of its own
@pytest.mark.parametrize("Nx", [32768, 32769, 40001])
def test_profiles_of_wide_channels(Nx):
    """C_l of every column from the densities of the same state with the library's
    mass ratios (FP32), a few roundings of FP64; the ends hold the boundary values."""
    p = workloads.preset("heli_argon_320x16", N=4, N_x=Nx, theta=1.2, Kn_out=0.3, C_l_out=0.4)
    g = binding.LbmMix(**p)
    g.init()
    g.step(2)
    s, m = g.separation(), g.moments()
    low = min(p["m_a"], p["m_b"])
    n = {k: m["rho_" + k].sum(axis=0) * float(np.float32(low / p["m_" + k])) for k in "ab"}
    light = "a" if p["m_a"] < p["m_b"] else "b"
    ref = (n[light] / (n["a"] + n["b"]))[1:-1]
    assert np.abs(s["Cl_profile"][1:-1] - ref).max() < 1e-13
    assert [s["Cl_profile"][0], s["Cl_profile"][-1]] == [p["C_l"], 0.4]
    assert s["CL"] == (p["C_l"] - s["Cl_profile"][s["x_min"]]) / p["C_l"]


def _us(f):
    best = math.inf
    for _ in range(7):
        t = time.perf_counter()
        f()
        best = min(best, time.perf_counter() - t)
    return 1e6 * best


def test_reading_a_wide_profile_takes_the_length_of_a_copy():
    torch = pytest.importorskip("torch")
    g = binding.LbmMix(**workloads.preset("heli_argon_320x16", N=4, N_x=1000000))
    g.init()
    g.step(1)
    d = torch.empty(1000000, dtype=torch.float64, device="cuda")
    assert _us(g.separation) < 2.0 * _us(d.cpu) + 100.0
