"""The autotuner keeps the collision CTAs per SM that were set when every value it
tries is the same launch (FP32: one CTA per SM is resident)."""
import pytest

from paper_2103_12194_gb300 import inputs

from .test_gpu_small import slpic  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_sm", [1, 3, 16])
def test_equal_collision_launches_do_not_compete(slpic, per_sm):  # noqa: F811
    spec = inputs.gap_spec(n_cells=64, V=100.0, pd_torr_cm=1.0, field_mode=0, charge_shift=20)
    for _ in range(3):
        sim = slpic.Simulation(1)
        sim.configure(0, spec, capacity=(1 << 16, 1 << 16))
        sim.seed(0, 0, 2000, slpic.SEED_GAP, e_lo=0.1, e_hi=5.0)
        sim.set_launch_shape(sim.launch_shape()[0], per_sm)
        warps, cc = sim.autotune(4)
        assert cc == per_sm and sim.launch_shape() == (warps, cc)
        sim.close()
