"""Electrons emitted at the cathode are appended in the order of the ions that
emitted them, over stores of less than one, one and several collision items
of 256 ion tiles, few or many emissions in a tile."""
import numpy as np
import pytest

from paper_2103_12194_gb300 import inputs

from .test_gpu_small import slpic  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("n", [1, 127, 128, 33 * 128 + 1, 256 * 128, 256 * 128 + 1, 600 * 128 + 5])
@pytest.mark.parametrize("share", [0.002, 0.3, 1.0])
def test_emitted_electrons_follow_their_ions(slpic, n, share, precision):  # noqa: F811
    spec = inputs.gap_spec(n_cells=32, V=100.0, pd_torr_cm=0.0, gamma_se=1.0, field_mode=0,
                           charge_shift=20)
    rng = np.random.default_rng(n)
    real = np.float64 if precision == 64 else np.float32
    out = rng.random(n) < share
    out[-1] = True
    m = {"cell": np.where(out, 0, 20).astype(np.int32), "off": np.full(n, 0.25, real),
         "vx": np.where(out, -2 * spec["d"] / spec["n_cells"] / spec["dt"], 0.0).astype(real),
         "vy": np.zeros(n, real), "vz": np.zeros(n, real),
         "wj": (1 + rng.random(n)).astype(real), "id": np.arange(n, dtype=np.uint32)}
    sim = slpic.Simulation(1, precision=precision)
    sim.configure(0, spec, capacity=(n + 128, n))
    sim.load(0, 1, m)
    sim.step(1)
    e = sim.particles(0, 0)
    # (an ion emits when a uniform number below 1 is below the yield of 1)
    assert np.array_equal(e["wj"], m["wj"][out])
    assert np.array_equal(e["id"] & 0x7FFFFFFF, np.arange(out.sum()))
    assert np.all(e["id"] >> 31 == 1) and not e["cell"].any() and not e["vx"].any()
    assert np.array_equal(sim.particles(0, 1)["id"], m["id"][~out])
    sim.close()
