"""lbm_mix_tune_rows with the library's own list: the default schedule is one of
its candidates, on channels of the step kernel too."""
import pytest

from paper_1603_08221_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,N,Nx", [(binding.LBM_FP32, 130, 5001), (binding.LBM_BF16, 130, 5001),
                                          (binding.LBM_FP32, 40, 700)])
def test_the_default_schedule_is_a_candidate(storage, N, Nx):
    p = workloads.preset("heli_argon_320x16", N=N, N_x=Nx, theta=1.2, Kn_out=0.3, storage=storage)
    g = binding.LbmMix(**p)
    g.init()
    best = g.tune_rows(steps=3)
    assert g.steps == 8 * (3 + 2)
    nmax = (N + 7) // 8 * 8
    assert best in {0} | {min(r, nmax) for r in (64, 72, 80, 88, 96, 112, 128)}


def test_the_default_schedule_is_returned_as_what_sets_it():
    """On a small channel several steps per launch are the fastest by far."""
    p = workloads.preset("heli_argon_320x16")
    g = binding.LbmMix(**p)
    g.init()
    assert g.tune_rows(steps=20) == 0
    assert g.tune_rows([8, 16], steps=3) in (8, 16)
