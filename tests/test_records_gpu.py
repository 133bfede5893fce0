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


# calls of one, two and three steps, of channels on both sides of the line
# between single steps by tiles and by the step kernel, and of sweeps
@pytest.mark.parametrize("N,Nx", [(16, 2048), (16, 2049), (8, 8263), (8, 40000), (2, 100000)])
def test_short_calls_take_no_longer_than_the_step_kernel(N, Nx):
    """Narrow channels take two launches where the step kernel takes one, a wide
    one nothing beyond it (its timing's spread: a third and 5 us)."""
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.2, Kn_out=0.3)
    slack = 2.0 if Nx <= 2048 else 4.0 / 3.0
    assert us_per_call(p, 0) < slack * us_per_call(p, 8 * ((N + 7) // 8)) + 5.0


@pytest.mark.parametrize("N,Nx", [(8, 2049), (16, 4000), (64, 3000)])
def test_wide_channels_split_over_calls_in_any_way(N, Nx):
    """The same populations whichever kernel takes a step, and the records to the
    rounding of their sums."""
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, diag_every=4, theta=1.2, Kn_out=0.3)
    total, runs = 40, []
    for rows, split in ((0, [40]), (0, [1] * 40), (0, [2, 3, 4, 5, 6, 7, 13]), (8, [40])):
        g = binding.LbmMix(**p)
        g.set_rows_per_block(rows)
        g.init()
        for n in split:
            g.step(n)
        assert g.steps == total
        runs.append(g)
    ref = runs[0]
    h = ref.history()
    assert len(h) == 10
    for g in runs[1:]:
        assert np.array_equal(g.get_post_state_f64()[..., 1:-1],
                              ref.get_post_state_f64()[..., 1:-1])
        m, mr = g.moments(), ref.moments()
        assert all(np.array_equal(m[k], mr[k]) for k in m)
        assert np.abs(g.history(1)[0, 6:8] / h[-1, 6:8] - 1).max() <= 2.0 ** -34
    assert np.array_equal(runs[3].history()[:, 0], h[:, 0])


@pytest.mark.parametrize("count,N,Nx,extra", [(8, 32, 400, dict(x_periodic=1)), (3, 20, 700, {}),
                                              (52, 20, 700, {})])
@pytest.mark.parametrize("split", [[1] * 12, [2] * 6, [3, 1, 2, 6]])
def test_sweeps_by_short_calls(count, N, Nx, extra, split):
    params = [workloads.preset("heli_argon_320x16", N=N, N_x=Nx + q % 2, theta=1.2 + 0.01 * q,
                               Kn_out=0.3, **extra) for q in range(count)]
    f0 = workloads.random_post_state(N, Nx, seed=4, lo=0.099, hi=0.101)
    f0[:, 0] *= 4.0
    sw, lone = binding.LbmSweep(params), {}
    sw.init()
    for q in (0, count - 1):
        lone[q] = g = binding.LbmMix(**params[q])
        g.init()
    if extra:
        for g in [sw.instance(0), lone[0]]:
            g.set_post_state(f0.astype(np.float32))
    for n in split:
        sw.step(n)
        for g in lone.values():
            g.step(n)
    for q, g in lone.items():
        a, b = sw.instance(q), g
        assert a.steps == b.steps == 12
        cols = slice(None) if extra else slice(1, -1)
        assert np.array_equal(a.get_post_state_f64()[..., cols], b.get_post_state_f64()[..., cols])
        assert np.abs(a.history(1)[0, 6:8] / b.history(1)[0, 6:8] - 1).max() <= 2.0 ** -34
