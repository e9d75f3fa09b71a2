"""What the host knows of a context's state: it must not go stale when steps
run in a graph that the caller captured, when markers are appended with and
without steps in between, or when the stream changes."""
import ctypes

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


@pytest.mark.parametrize("call", ["set_voltage", "seed", "count", "tallies", "field", "charge",
                                  "reset_counters", "history"])
def test_refused_while_captured(slpic, call):  # noqa: F811
    """Calls that answer on the host, or change what the host holds, are
    refused while their stream is captured, also when the state is known; the
    context is as before after it."""
    import torch
    cuda = ctypes.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    sim, plain = make(slpic, 1, stream), make(slpic, 1)
    for s in (sim, plain):
        s.step(3)
        s.count(0, 0)  # the state is known from here
    args = {"set_voltage": (0, 300.0), "seed": (0, 0, 5, slpic.SEED_REST),
            "count": (0, 0), "charge": (0, 0)}
    graph, handle = ctypes.c_void_p(), ctypes.c_void_p(stream.cuda_stream)
    assert cuda.cuStreamBeginCapture_v2(handle, 1) == 0  # this thread's calls alone
    try:
        with pytest.raises(slpic.SlpicError):
            getattr(sim, call)(*args.get(call, (0,)))
    finally:
        assert cuda.cuStreamEndCapture(handle, ctypes.byref(graph)) != 0  # invalidated
    for s in (sim, plain):
        s.set_voltage(0, 300.0)
        s.step(2)
    same(sim, plain)
    sim.close()
    plain.close()


def test_uploads_arrive_before_steps_on_other_streams(slpic):  # noqa: F811
    """Steps captured on the context's stream and replayed on another one find
    what the calls before them have set, those before the capture too; a stream
    that is destroyed may be replaced."""
    import torch
    cuda = ctypes.CDLL("libcuda.so.1")
    own = ctypes.c_void_p()
    sim, plain = make(slpic, 0), make(slpic, 0)
    sim.synchronize()
    assert cuda.cuStreamCreate(ctypes.byref(own), 1) == 0
    sim.set_stream(own.value)
    for s in (sim, plain):
        s.set_voltage(0, 280.0)
    assert cuda.cuStreamSynchronize(own) == 0 and cuda.cuStreamDestroy_v2(own) == 0
    stream, other = torch.cuda.Stream(), torch.cuda.Stream()
    sim.set_stream(stream)
    graph = torch.cuda.CUDAGraph()
    for s in (sim, plain):
        s.seed(0, 0, 300, slpic.SEED_REST)
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        sim.step(1)
    with torch.cuda.stream(other):
        for V in (250.0, 350.0, 150.0):
            sim.set_voltage(0, V)
            graph.replay()
            other.synchronize()
            plain.set_voltage(0, V)
            plain.step(1)
            same(sim, plain)
    sim.close()
    plain.close()
