"""A store of a batch that overflows: the kernels' CTAs stop as one while the
error is set, the step ends, and freshly loaded markers step as in a new
context."""
import numpy as np
import pytest

from paper_2103_12194_gb300 import inputs

from .test_gpu_parity import mixed_state
from .test_gpu_small import slpic  # noqa: F401

pytestmark = pytest.mark.gpu

N = 12


def make(slpic):  # noqa: F811
    sim = slpic.Simulation(N)
    specs = [inputs.gap_spec(n_cells=64 + 16 * i, V=300.0, pd_torr_cm=40.0, gamma_se=0.3,
                             field_mode=i % 2, seed=50 + i, instance=i) for i in range(N)]
    for i, spec in enumerate(specs):
        sim.configure(i, spec, capacity=(1 << 15, 1 << 15) if i else (4000, 4000))
    return sim, specs


def load(sim, specs, n):
    for i, spec in enumerate(specs):
        for s, m in enumerate(mixed_state(spec, n, n // 2, seed=3 * i)):
            sim.load(i, s, m)


def test_one_store_of_a_batch_overflows(slpic):  # noqa: F811
    sim, specs = make(slpic)
    for _ in range(20):
        load(sim, specs, 4000)  # the first instance's store is full
        with pytest.raises(slpic.SlpicError) as e:
            sim.step(2)
            sim.synchronize()
        assert e.value.code == slpic.ERR_CAPACITY
        sim.clear_error()
    fresh, _ = make(slpic)
    for s in (sim, fresh):
        load(s, specs, 1000)
        for i in range(N):
            s.reset_counters(i)
        s.step(2)
    for i in range(N):
        assert np.array_equal(sim.history(i), fresh.history(i)), i
        for s in (0, 1):
            assert np.array_equal(sim.charge(i, s), fresh.charge(i, s)), (i, s)
            a, b = sim.particles(i, s), fresh.particles(i, s)
            for k in a:
                assert np.array_equal(a[k], b[k]), (i, s, k)
    sim.close()
    fresh.close()
