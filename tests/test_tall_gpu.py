"""FP32 channels of more rows than the tiles and the eight-lane column sums take:
the sums of the end columns behind the density correction (Eq. rho2) by whole
CTAs."""
import math
import time

import numpy as np
import pytest

from paper_1603_08221_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


# both sides of the line at 512 rows; a last round of rows that is short, full
# and one over for 256 threads; both ends in one strip and in two, the columns
# N_x - 2 and N_x - 3 in one strip or in two (N_x = 98)
@pytest.mark.parametrize("N", [512, 513, 767, 768, 1025, 2600])
@pytest.mark.parametrize("Nx", [7, 98])
def test_end_columns_of_tall_channels(N, Nx):
    """The stored column sums against exact sums of the densities of the same
    state: the nodes' sums of deviations are added as pairs of floats and cut at
    2^-48 of the column's sum, so 2^-44 of it covers the additions' errors too.
    And the same bits under every schedule and split of the calls."""
    torch = pytest.importorskip("torch")
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.3, Kn_out=0.3, diag_every=3)
    states = []
    for rows, split in ((0, [9]), (0, [1] * 9), (64, [4, 5]), (512, [9])):
        g = binding.LbmMix(**p)
        g.set_rows_per_block(rows)
        g.init()
        for n in split:
            g.step(n)
        g.sync()
        states.append(g.get_post_state_f64()[..., 1:-1])
        cs = torch.as_tensor(g.device_views()["colsum"], device="cuda").cpu().numpy()
        m = g.moments()
        for x in (1, 2, Nx - 3, Nx - 2):
            for sp, name in enumerate(("rho_a", "rho_b")):
                exact = math.fsum(m[name][:, x])
                assert abs(cs[sp, x] - exact) <= 2.0 ** -44 * exact, (rows, x, name)
    assert np.isfinite(states[0]).all()
    for f in states[1:]:
        assert np.array_equal(f, states[0])


def _us_per_step(p):
    g = binding.LbmMix(**p)
    g.init()
    g.step(20)
    g.sync()
    best = math.inf
    for _ in range(5):
        t = time.perf_counter()
        g.step(20)
        g.sync()
        best = min(best, time.perf_counter() - t)
    return 1e6 * best / 20


def test_end_columns_do_not_dominate_a_step():
    """A step with pressure ends sums four columns of 64 that a periodic one does
    not, each read once more, and in one CTA: they may cost a launch's length
    (some 10 us) and no more than the rest of the step."""
    p = workloads.preset("heli_argon_320x16", N=16384, N_x=64, theta=1.2, Kn_out=0.3,
                         diag_every=1000)
    assert _us_per_step(p) < 2.0 * _us_per_step(dict(p, x_periodic=1)) + 10.0
