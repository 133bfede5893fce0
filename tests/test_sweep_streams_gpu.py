"""The handles of a sweep keep streams of their own: a call on one waits for its
own work, and the sweep's common launches come after what calls left there."""
import time

import numpy as np
import pytest

from paper_1603_08221_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


def test_a_borrowed_handle_waits_for_its_own_work():
    """9000 steps of one channel take some 20 ms of the GPU, issuing them a few;
    a step of another waits for the latter alone."""
    sw = binding.LbmSweep([workloads.preset("paper_case2_700x20")] * 2)
    sw.init()
    a, b = sw.instance(0), sw.instance(1)
    for h in (a, b):
        h.step(100)
        h.sync()
    t0 = time.perf_counter()
    a.step(9000)
    b.step(1)
    b.sync()
    tb = time.perf_counter() - t0
    a.sync()
    ta = time.perf_counter() - t0
    assert tb < 0.5 * ta


@pytest.mark.parametrize("N,Nx", [(20, 700), (130, 900)])
def test_a_sweep_comes_after_calls_on_its_handles(N, Nx):
    """Calls that return before their work is done (init, step, rereference) and
    calls of the sweep, in turn without a wait: a lone handle's populations."""
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.2, Kn_out=0.3)
    sw = binding.LbmSweep([p] * 3)
    ref = binding.LbmMix(**dict(p, reref_every=0))
    sw.init()
    ref.init()
    for n in (2000, 7, 1):
        sw.instance(1).step(n)
        sw.step(11)
        sw.instance(1).rereference()
        sw.run_to_steady(1e-14, 4, 2)
        for k in (n, 11):
            ref.step(k)
        ref.rereference()
        ref.step(2)
        ref.step(2)
    sw.instance(1).init()
    sw.step(5)
    sw.instance(1).step(300)
    ref.init()
    ref.step(305)
    assert np.array_equal(sw.instance(1).get_post_state_f64()[..., 1:-1],
                          ref.get_post_state_f64()[..., 1:-1])
