"""States that are none of a gas are reported: a node where a species density is
zero or negative gives non-finite rates (psi and its square roots have no value
there), so the step's record and the node's fields are non-finite, in every
storage type and schedule, whichever species and reading of lambda_sigma."""
import numpy as np
import pytest

from paper_1603_08221_gb300 import binding, workloads

pytestmark = pytest.mark.gpu

SPECIES = {"a": (0,), "b": (1,), "both": (0, 1)}


def _state(g, species, factor):
    f = np.asarray(g.get_post_state(), dtype=np.float32)
    for sp in SPECIES[species]:
        f[sp, :, 6:11, 30:36] *= np.float32(factor)
    return f


@pytest.mark.parametrize("species", list(SPECIES))
@pytest.mark.parametrize("factor", [-1.0, -1e-3])
@pytest.mark.parametrize("storage,rows,lam", [(binding.LBM_FP32, 0, 0), (binding.LBM_FP32, 0, 1),
                                              (binding.LBM_FP32, 8, 0), (binding.LBM_FP32, 16, 1),
                                              (binding.LBM_BF16, 0, 0)])
def test_negative_densities_are_reported(species, factor, storage, rows, lam):
    p = workloads.preset("heli_argon_320x16", N=16, N_x=64, storage=storage, lambda_pressure=lam)
    g = binding.LbmMix(**p)
    g.init()
    g.step(3)
    g.set_post_state(_state(g, species, factor))
    g.set_rows_per_block(rows)
    g.step(1)
    with pytest.raises(binding.LbmError) as e:
        g.separation()
    assert e.value.status == binding.LBM_ENONFINITE
    m = g.moments()
    assert not any(np.isfinite(m[k][8, 33]) for k in ("ua_x", "ua_y", "ub_x", "ub_y"))
    assert not np.isfinite(g.get_post_state_f64()[:, 1:, 8, 33]).any()


@pytest.mark.parametrize("species", list(SPECIES))
@pytest.mark.parametrize("factor", [-1.0, 0.0])
@pytest.mark.parametrize("steps", [0, 1])
@pytest.mark.parametrize("storage", [binding.LBM_FP32, binding.LBM_FP16])
def test_volume_flow_through_a_node_without_gas_is_refused(species, factor, steps, storage):
    """As the fields are: Eq. rhou divides by each species' density."""
    p = workloads.preset("heli_argon_320x16", N=16, N_x=64, storage=storage)
    g = binding.LbmMix(**p)
    g.init()
    g.step(3)
    g.set_post_state(_state(g, species, factor))
    g.step(steps)
    assert np.isnan(g.moments()["ua_x"][8, 33] + g.moments()["ub_x"][8, 33])
    with pytest.raises(binding.LbmError) as e:
        g.volume_flow(33)
    assert e.value.status == binding.LBM_ENONFINITE
    assert np.isfinite(g.volume_flow(50))
