"""The records' sums over columns, row blocks and strips against FP64 sums of the
populations, over row blocks of every kind (one, several, a short last one),
widths around the strips, and storage types.

Tolerances, derived.  Between schedules the terms are the same and only their
order differs: every partial sum is a pair of floats, exact to 2^-44 of the
largest partial sum, of which there are fewer than 2^10 in a row, so 2^-34 of the
sums of the terms' magnitudes.  Against the populations: a node's density and
momentum are formed from nine FP32 deviations and the collision conserves them to
rounding, fewer than 64 roundings of 2^-24 of the magnitudes, with 16-bit storage
one more, stochastic, of 2^-7 (BF16) or 2^-10 (FP16) of each stored deviation;
deviations and reference add up to at most twice the populations' magnitudes."""
import math

import numpy as np
import pytest

from paper_1603_08221_gb300 import binding, workloads

pytestmark = pytest.mark.gpu

STORED = {binding.LBM_FP32: 0.0, binding.LBM_BF16: 2.0 ** -7, binding.LBM_FP16: 2.0 ** -10}


@pytest.mark.parametrize("storage", list(STORED))
@pytest.mark.parametrize("N,Nx,periodic", [(3, 6, 0), (17, 33, 0), (64, 98, 0), (131, 257, 0),
                                           (40, 64, 1)])
def test_record_sums(storage, N, Nx, periodic):
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.2, Kn_out=0.3, storage=storage,
                         x_periodic=periodic, wall=periodic, diag_every=1)
    f0 = workloads.random_post_state(N, Nx, seed=4, lo=0.099, hi=0.101).astype(np.float32)
    cols = slice(0, Nx) if periodic else slice(1, Nx - 1)
    first = None
    for rows in (8, 16, 64, 512):
        g = binding.LbmMix(**p)
        g.set_post_state(f0)
        g.set_rows_per_block(rows)
        g.step(1)
        rec = g.history(1)[0]
        f = np.asarray(g.get_post_state_f64(), dtype=np.float64).reshape(2, 9, N, Nx)[..., cols]
        total = f.sum(axis=(1, 2, 3))
        tol = 2 * (64 * 2.0 ** -24 + STORED[storage]) * np.abs(f).sum(axis=(1, 2, 3))
        assert np.all(np.abs(rec[6:8] - total) <= tol), rows
        n = f.shape[-1]
        if first is None:
            first = rec
        assert np.all(np.abs(rec[6:8] - first[6:8]) <= 2.0 ** -34 * total)
        assert np.all(np.abs(rec[3:5] - first[3:5]) <= 2.0 ** -34 * total / n)
        assert abs(rec[1] - first[1]) <= 2.0 ** -30 and abs(rec[2] - first[2]) <= 2.0 ** -30


# Shapes of the step kernel whose recorded steps take other row blocks than the
# steps between them (more rows; one block where the others have several; all
# of the rows in either).  FP32 populations are the same bits under every
# schedule, 16-bit ones as far as the sums behind the density correction, which
# differ by less than 2^-40, round to the same FP32 factors.
@pytest.mark.parametrize("storage,N,Nx", [(binding.LBM_FP32, 130, 5001), (binding.LBM_FP32, 57, 9000),
                                          (binding.LBM_BF16, 8, 64), (binding.LBM_BF16, 57, 98),
                                          (binding.LBM_FP16, 131, 257)])
def test_default_schedule_of_recorded_steps(storage, N, Nx):
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.2, Kn_out=0.3, storage=storage,
                         diag_every=2)
    f0 = workloads.random_post_state(N, Nx, seed=4, lo=0.099, hi=0.101).astype(np.float32)
    out = []
    for rows in (0, 16):
        g = binding.LbmMix(**p)
        g.set_post_state(f0)
        g.set_rows_per_block(rows)
        g.step(5)
        out.append((np.asarray(g.get_post_state_f64()), g.history()[-3:]))
    (fa, ra), (fb, rb) = out
    # (the random state's outlet column turns non-finite within the five steps on
    # the largest shapes, under every schedule alike)
    assert np.array_equal(fa, fb, equal_nan=True)
    np.testing.assert_allclose(ra[:, 6:8], rb[:, 6:8], rtol=2.0 ** -34, atol=0.0, equal_nan=True)


# The stored sums of a column's densities against exact sums of the densities
# of the same state (the moment fields hold reference plus deviation, exact to
# 2^-53): the nodes' deviations are added as pairs of floats, exact but for the
# sum of the errors (2^-48 of the terms), and the total is cut at 2^-48, so 2^-44
# of it covers either, and N additions of the fields' last bits.
@pytest.mark.parametrize("N,Nx", [(9, 40), (20, 700), (37, 1001), (64, 500), (130, 300)])
@pytest.mark.parametrize("rows", [0, 8, 64])
def test_column_sums_are_exact_sums(N, Nx, rows):
    torch = pytest.importorskip("torch")
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.3, Kn_out=0.3)
    g = binding.LbmMix(**p)
    g.set_rows_per_block(rows)
    # deviations as large as the densities, of either sign within a column
    g.set_post_state(workloads.random_post_state(N, Nx, seed=N).astype(np.float32))
    g.step(1)
    g.sync()
    cs = torch.as_tensor(g.device_views()["colsum"], device="cuda").cpu().numpy()
    m = g.moments()
    for x in range(1, Nx - 1):
        for sp, name in enumerate(("rho_a", "rho_b")):
            exact = math.fsum(m[name][:, x])
            assert abs(cs[sp, x] - exact) <= 2.0 ** -44 * exact, (x, name)


def _disturbed(g, amplitude, seed):
    """The initial equilibrium, every population changed by its own factor."""
    g.init()
    f = np.asarray(g.get_post_state(), dtype=np.float64)
    rng = np.random.default_rng(seed)
    return (f * (1.0 + amplitude * rng.uniform(-1.0, 1.0, f.shape))).astype(np.float32)


# The shapes of the test above, from a state that stays finite, so that every
# record counts, and the mass flows beside the totals: 2^-34 of the sums of the
# magnitudes (see the top), which for the momenta are at most the masses.
@pytest.mark.parametrize("storage,N,Nx", [(binding.LBM_FP32, 130, 5001), (binding.LBM_FP32, 57, 9000),
                                          (binding.LBM_BF16, 8, 64), (binding.LBM_BF16, 57, 98),
                                          (binding.LBM_FP16, 131, 257)])
def test_recorded_steps_of_a_finite_state(storage, N, Nx):
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.2, Kn_out=0.3, storage=storage,
                         diag_every=2)
    out = []
    for rows in (0, 16):
        g = binding.LbmMix(**p)
        g.set_post_state(_disturbed(g, 0.01, seed=N))
        g.set_rows_per_block(rows)
        g.step(5)
        out.append((np.asarray(g.get_post_state_f64())[..., 1:-1], g.history()))
    (fa, ra), (fb, rb) = out
    assert len(ra) == len(rb) == 3
    assert all(np.isfinite(v).all() for v in (fa, fb, ra, rb))
    assert np.array_equal(fa, fb)
    total = rb[:, 6:8]
    assert np.all(np.abs(ra[:, 6:8] - total) <= 2.0 ** -34 * total)
    assert np.all(np.abs(ra[:, 3:5] - rb[:, 3:5]) <= 2.0 ** -34 * total / (Nx - 2))
    assert np.all(np.abs(ra[:, 1:3] - rb[:, 1:3]) <= 2.0 ** -30)
