"""What the host knows of a context's state: it must not go stale when steps
run in a graph that the caller captured, when markers are appended with and
without steps in between, or when the stream changes."""
import numpy as np
import pytest

from paper_2103_12194_gb300 import inputs

from .test_gpu_parity import mixed_state, slpic  # noqa: F401

pytestmark = pytest.mark.gpu


def make(slpic, field_mode, stream=None):  # noqa: F811
    spec = inputs.gap_spec(n_cells=64, V=300.0, pd_torr_cm=5.0, gamma_se=0.3,
                           field_mode=field_mode, charge_shift=24)
    sim = slpic.Simulation(1, stream=stream)
    sim.configure(0, spec, capacity=(1 << 15, 1 << 15))
    for s, m in enumerate(mixed_state(spec, 3000, 1000, seed=4)):
        sim.load(0, s, m)
    return sim


def same(a, b):
    for s in (0, 1):
        assert a.count(0, s) == b.count(0, s)
        x, y = a.particles(0, s), b.particles(0, s)
        for k in x:
            assert np.array_equal(x[k], y[k]), (s, k)
        assert np.array_equal(a.charge(0, s), b.charge(0, s))
    assert np.array_equal(a.history(0), b.history(0)) and a.tallies(0) == b.tallies(0)


def test_steps_replayed_by_a_caller(slpic):  # noqa: F811
    """Steps captured into the caller's graph: each replay advances the
    context, and every read sees it."""
    import torch
    stream = torch.cuda.Stream()
    sim, plain = make(slpic, 1, stream), make(slpic, 1)
    sim.count(0, 0)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        sim.step(2)
    for _ in range(3):
        with torch.cuda.stream(stream):
            graph.replay()
        plain.step(2)
        same(sim, plain)
    sim.step(1)
    plain.step(1)
    same(sim, plain)
    sim.close()
    plain.close()


@pytest.mark.parametrize("field_mode", [0, 1])
def test_appending_with_and_without_steps(slpic, field_mode):  # noqa: F811
    """seed after a load, after a seed, after steps and after emptying the
    store, with a change of stream on the way, equals the same calls with a
    synchronisation and a read after each."""
    import torch
    one, two = make(slpic, field_mode), make(slpic, field_mode)

    def both(f, settle=True):
        for sim in (one, two):
            f(sim)
        if settle:
            two.synchronize()
            two.particles(0, 0)

    none = {k: np.empty(0, slpic.DTYPES.get(k, np.float32)) for k in slpic.FIELDS}
    for k, n in enumerate((1, 127, 500)):
        both(lambda s: s.seed(0, 0, n, slpic.SEED_GAP, e_lo=1.0, e_hi=50.0))
        both(lambda s: s.seed(0, 1, n, slpic.SEED_THERMAL))
        both(lambda s: s.step(k))
        if k == 1:
            one.set_stream(torch.cuda.Stream())
            both(lambda s: s.load(0, 0, none))
            both(lambda s: s.reset_counters(0))
            both(lambda s: s.set_voltage(0, 250.0))
    same(one, two)
    one.close()
    two.close()
