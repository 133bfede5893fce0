"""Several steps per launch (lbm_tile_kernel: tiles of whole columns with
halos in shared memory), the default of small FP32 channels.

Against the step kernel (a row count set by the caller) the densities are held
to 1e-6 and the velocities to 1e-5 of their largest, the bounds the schedules
of the step kernel are held to; and since every schedule adds the columns
behind the ends' density correction in one order, the populations are the same
bits under all of them, however a run is split over calls and whether a channel
runs alone or in a sweep."""
import numpy as np
import pytest

from paper_1603_08221_gb300 import binding, workloads

pytestmark = pytest.mark.gpu

RTOL = 1e-6

# rows and columns around the kernel's edges: two rows (no inner row), odd and
# even row counts (the padded column), channels narrower than a halo, one
# tile, one more column than a multiple of the SMs, several nodes per thread
SIZES = [(2, 5, 9), (3, 4, 8), (5, 7, 20), (8, 33, 31), (16, 155, 40), (17, 307, 40),
         (31, 1000, 30), (64, 700, 30), (65, 460, 30), (100, 300, 20)]


def _close(g, ref):
    m, mr = g.moments(), ref.moments()
    scale = max(np.abs(mr["ua_x"]).max(), np.abs(mr["ub_x"]).max())
    for k in m:
        tol = RTOL * np.abs(mr[k]).max() if k.startswith("rho") else 10 * RTOL * scale + 3e-8
        assert np.abs(m[k] - mr[k]).max() <= tol, k


@pytest.mark.parametrize("N,Nx,steps", SIZES)
@pytest.mark.parametrize("extra", [dict(), dict(x_periodic=1),
                                   dict(wall=binding.LBM_WALL_BSR, r_form=binding.LBM_R_SECOND,
                                        lambda_pressure=1, C_l_out=0.4)])
def test_tiles_against_the_step_kernel(N, Nx, steps, extra):
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.2, Kn_out=0.3, **extra)
    alpha = workloads.random_accommodation(Nx, seed=N, spread=0.2)
    f = workloads.random_post_state(N, Nx, seed=3, lo=0.099, hi=0.101)
    w = np.ones((2, 9, N, Nx))
    w[:, 0] = 4.0  # close to an equilibrium, so that few-row channels stay tame
    runs = []
    for rows in (0, 8):
        g = binding.LbmMix(diag_every=3, **p)
        g.set_rows_per_block(rows)
        g.set_accommodation_field(alpha)
        if extra.get("x_periodic"):
            g.set_post_state((f * w).astype(np.float32))
        else:
            g.init()
        g.step(steps)
        runs.append(g)
    _close(*runs)
    h, hr = runs[0].history(), runs[1].history()
    assert h.shape == hr.shape and np.array_equal(h[:, 0], hr[:, 0])
    assert np.abs(h[:, 6:] / hr[:, 6:] - 1).max() < RTOL
    s, sr = runs[0].separation(), runs[1].separation()
    assert np.abs(s["Cl_profile"] - sr["Cl_profile"]).max() < RTOL


@pytest.mark.parametrize("N,Nx", [(16, 320), (21, 700), (64, 500)])
@pytest.mark.parametrize("diag_every,reref", [(1, 0), (4, 0), (100, 7)])
def test_calls_split_in_any_way_give_the_same_bits(N, Nx, diag_every, reref):
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, diag_every=diag_every,
                         reref_every=reref)
    total = 60
    runs = []
    for split in ([60], [1] * 60, [2, 3, 5, 7, 11, 13, 19]):
        g = binding.LbmMix(**p)
        g.init()
        for n in split:
            g.step(n)
        assert g.steps == total
        runs.append(g)
    for g in runs[1:]:
        assert np.array_equal(g.get_post_state_f64()[..., 1:-1],
                              runs[0].get_post_state_f64()[..., 1:-1])
        m, mr = g.moments(), runs[0].moments()
        assert all(np.array_equal(m[k], mr[k]) for k in m)
        assert np.array_equal(g.history(1)[0, 1:], runs[0].history(1)[0, 1:])


def test_captured_steps_replay():
    """Steps captured into a CUDA graph replay what direct calls run."""
    torch = pytest.importorskip("torch")
    p = workloads.preset("paper_case2_700x20")
    runs = []
    for capture in (False, True):
        stream = torch.cuda.Stream()
        g = binding.LbmMix(stream=stream, **p)
        g.init()
        g.step(2)
        g.sync()
        if capture:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                g.step(24)
            with torch.cuda.stream(stream):
                graph.replay()
                graph.replay()
        else:
            g.step(24)
            g.step(24)
        g.sync()
        runs.append((g.get_post_state_f64(), g.history()))
    assert np.array_equal(runs[0][0], runs[1][0])
    assert np.array_equal(runs[0][1], runs[1][1])


def test_tuning_keeps_the_default_where_it_is_fastest():
    """The library's own candidate list includes the several-steps schedule
    (the fastest by far on a small channel), a caller's list does not."""
    p = workloads.preset("heli_argon_320x16")
    g = binding.LbmMix(**p)
    g.init()
    g.tune_rows(steps=20)
    g.init()
    g.step(50)
    ref = binding.LbmMix(**p)
    ref.init()
    ref.step(50)
    assert np.array_equal(g.get_post_state_f64(), ref.get_post_state_f64())
    assert g.tune_rows([8, 16], steps=3) in (8, 16)


# column counts around the strip edges of the end columns: N_x - 2 and N_x - 3
# in one strip of 32 columns or in two (N_x = 98), both ends in one strip
@pytest.mark.parametrize("N,Nx", [(20, 100), (33, 98), (9, 97), (64, 99), (130, 66), (12, 20)])
@pytest.mark.parametrize("extra", [dict(), dict(wall=binding.LBM_WALL_BSR, C_l_out=0.4)])
def test_populations_are_the_same_bits_under_every_schedule(N, Nx, extra):
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.3, Kn_out=0.3, **extra)
    alpha = workloads.random_accommodation(Nx, seed=1, spread=0.2)
    states = []
    for rows, diag_every in ((0, 1), (0, 7), (8, 1), (8, 100), (24, 7), (64, 3)):
        g = binding.LbmMix(diag_every=diag_every, **p)
        g.set_rows_per_block(rows)
        g.set_accommodation_field(alpha)
        g.init()
        g.step(30)
        states.append(g.get_post_state_f64()[..., 1:-1])
    for f in states[1:]:
        assert np.array_equal(f, states[0])


@pytest.mark.parametrize("count,N,Nx", [(3, 20, 700), (60, 20, 300), (24, 64, 1000),
                                        (5, 130, 900)])
def test_sweeps_take_the_steps_of_lone_channels(count, N, Nx):
    """Few and many channels, small and tall ones: tiles or the batched step
    kernel, the populations are those of each channel on its own."""
    params = [workloads.preset("heli_argon_320x16", N=N, N_x=Nx + q % 3, theta=1.2 + 0.01 * q,
                               Kn_out=0.3) for q in range(count)]
    sw = binding.LbmSweep(params)
    sw.init()
    sw.step(7)
    sw.run_to_steady(1e-14, 20, 10)
    for q in (0, 1, count - 1):
        g = binding.LbmMix(**params[q])
        g.init()
        g.step(27)
        assert sw.instance(q).steps == 27
        assert np.array_equal(sw.instance(q).get_post_state_f64()[..., 1:-1],
                              g.get_post_state_f64()[..., 1:-1]), q
        a, b = sw.instance(q).separation(), g.separation()
        assert abs(a["CL"] - b["CL"]) < 1e-9 and a["x_min"] == b["x_min"]


@pytest.mark.parametrize("steps", [[9], [1, 8], [5, 2, 2]])
def test_sweeps_of_tiled_and_other_channels(steps):
    """Channels that qualify for tiles, of three row counts, among more others
    than one launch of the step kernel holds (32): each as on its own."""
    small = [dict(N=n, N_x=300 + 40 * q) for q, n in enumerate([16, 20, 20, 24, 16, 20])]
    tall = [dict(N=440 + 8 * (q % 3), N_x=60 + 7 * (q % 5)) for q in range(38)]
    params = [workloads.preset("heli_argon_320x16", theta=1.2 + 0.005 * q, Kn_out=0.3, **d)
              for q, d in enumerate(tall[:20] + small + tall[20:])]
    sw = binding.LbmSweep(params)
    sw.init()
    for n in steps:
        sw.step(n)
    for q in (0, 19, 20, 22, 25, 26, 40, len(params) - 1):
        g = binding.LbmMix(**params[q])
        g.init()
        for n in steps:
            g.step(n)
        assert sw.instance(q).steps == sum(steps)
        assert np.array_equal(sw.instance(q).get_post_state_f64()[..., 1:-1],
                              g.get_post_state_f64()[..., 1:-1]), q
