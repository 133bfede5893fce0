"""The records of channels that take several steps per launch: blocks of 256
columns each, up to 128 of them, folded by the last."""
import math
import time

import numpy as np
import pytest

from paper_1603_08221_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


# one block, a full and a short last one, as many as there are, more columns than
# they take in one pass; records of one step and of many
@pytest.mark.parametrize("N,Nx", [(4, 5), (9, 256), (9, 257), (16, 513), (4, 2049), (2, 32768),
                                  (2, 40001)])
@pytest.mark.parametrize("periodic", [0, 1])
def test_records_of_tiles_against_the_step_kernel(N, Nx, periodic):
    """The same node sums, as pairs of floats that are exact to 2^-44, added over
    the columns in another order in FP64: 2^-34 of the sums of the magnitudes, as
    between the step kernel's schedules; C_l and what is formed from it 2^-30."""
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.2, Kn_out=0.3,
                         x_periodic=periodic, diag_every=2)
    f0 = workloads.random_post_state(N, Nx, seed=4, lo=0.099, hi=0.101)
    f0[:, 0] *= 4.0  # close to an equilibrium
    recs, seps = [], []
    for rows in (0, 8):
        g = binding.LbmMix(**p)
        g.set_rows_per_block(rows)
        if periodic:
            g.set_post_state(f0.astype(np.float32))
        else:
            g.init()
        for n in (1, 1, 7, 4):
            g.step(n)
        recs.append(g.history())
        seps.append(g.separation())
    a, b = recs
    assert a.shape == b.shape and np.isfinite(a).all()
    assert np.array_equal(a[:, 0], b[:, 0])
    total = b[:, 6:8]
    assert np.all(np.abs(a[:, 6:8] - total) <= 2.0 ** -34 * total)
    assert np.all(np.abs(a[:, 3:5] - b[:, 3:5]) <= 2.0 ** -34 * total / (Nx if periodic else Nx - 2))
    assert np.all(np.abs(a[:, 1:3] - b[:, 1:3]) <= 2.0 ** -30)
    prof = np.abs(seps[0]["Cl_profile"] - seps[1]["Cl_profile"])
    assert prof.max() <= 2.0 ** -30
    xa, xb = seps[0]["x_min"], seps[1]["x_min"]
    assert xa == xb or abs(seps[0]["Cl_profile"][xa] - seps[0]["Cl_profile"][xb]) <= 2.0 ** -30


def us_per_call(p, rows, calls=30):
    """Calls of a single step, without a wait between them."""
    g = binding.LbmMix(**p)
    g.set_rows_per_block(rows)
    g.init()
    g.step(20)
    g.sync()
    best = math.inf
    for _ in range(5):
        t = time.perf_counter()
        for _ in range(calls):
            g.step(1)
        g.sync()
        best = min(best, time.perf_counter() - t)
    return 1e6 * best / calls


@pytest.mark.parametrize("N,Nx", [(8, 40000), (20, 20000), (2, 100000)])
def test_a_record_does_not_dominate_a_call_of_one_step(N, Nx):
    """The step kernel takes a step and its record in one launch; two launches may
    take some twice as long, but not a multiple that grows with the columns."""
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.2, Kn_out=0.3)
    assert us_per_call(p, 0) < 3.0 * us_per_call(p, 8 * ((N + 7) // 8)) + 5.0
