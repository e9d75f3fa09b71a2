"""The field of the Poisson solve around the blocks of nodes that it is formed
in, for gaps alone and side by side in one context, against the oracle; the
bars are those of test_poisson_matches_oracle."""
import numpy as np
import pytest

from paper_2103_12194_gb300 import inputs

from .test_gpu_parity import mixed_state, slpic  # noqa: F401

pytestmark = pytest.mark.gpu

CELLS = (2, 3, 1022, 1023, 1024, 1025, 2047, 2048, 5000)


def check(slpic, oracle_mod, cells, field_modes):  # noqa: F811
    sim = slpic.Simulation(len(cells))
    specs, states = [], []
    for k, (n, mode) in enumerate(zip(cells, field_modes)):
        spec = inputs.gap_spec(n_cells=n, V=300.0, pd_torr_cm=20.0, gamma_se=0.5,
                               field_mode=mode, charge_shift=16, instance=k)
        spec["dt"] = 0.0
        e, i = mixed_state(spec, 3000, 5000, seed=20 + k)
        for m in (e, i):
            m["cell"] = (np.arange(m["cell"].size) * 7 % n).astype(np.int32)
            m["wj"] *= np.float32(3e6)  # strong enough space charge to bend phi
        specs.append(spec)
        states.append((e, i))
        sim.configure(k, spec, capacity=(16384, 16384))
    for k, (e, i) in enumerate(states):
        sim.load(k, 0, e)
        sim.load(k, 1, i)
    sim.step(1)
    for k, spec in enumerate(specs):
        ref = oracle_mod.Oracle(spec, precision=32)
        ref.load(0, states[k][0])
        ref.load(1, states[k][1])
        ref.step(1)
        for s in (0, 1):
            assert np.array_equal(sim.charge(k, s), ref.charge(s)), (k, s)
        phi_g, E_g = sim.field(k)
        phi_r, E_r = ref.field()
        assert np.allclose(phi_g, phi_r, rtol=1e-10, atol=1e-10 * spec["V"]), k
        assert np.allclose(E_g, E_r, rtol=1e-8, atol=1e-8 * np.abs(E_r).max()), k
    sim.close()


def test_blocks_side_by_side(slpic, oracle_mod):  # noqa: F811
    check(slpic, oracle_mod, CELLS, [1] * len(CELLS))
    check(slpic, oracle_mod, CELLS, [k % 2 for k in range(len(CELLS))])


@pytest.mark.parametrize("n", CELLS)
def test_blocks_of_one_gap(slpic, oracle_mod, n):  # noqa: F811
    check(slpic, oracle_mod, (n,), (1,))
