"""Steps that the host has not waited for: replayed in a caller's graph after the
stores have changed, and in flight on a stream that the context leaves."""
import numpy as np
import pytest

from paper_2103_12194_gb300 import inputs

from .test_gpu_host_state import make, same
from .test_gpu_parity import mixed_state, slpic  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("field_mode", [0, 1])
def test_replays_after_the_stores_have_changed(slpic, field_mode):  # noqa: F811
    import torch
    stream = torch.cuda.Stream()
    spec = inputs.gap_spec(n_cells=64, V=300.0, pd_torr_cm=5.0, gamma_se=0.3,
                           field_mode=field_mode, charge_shift=24)
    sim, plain = make(slpic, field_mode, stream), make(slpic, field_mode)
    for s in (sim, plain):
        s.step(1)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        sim.step(1)

    def load(n, seed):
        def change(s):
            for sp, m in enumerate(mixed_state(spec, n, n // 2, seed=seed)):
                s.load(0, sp, m)
        return change

    for change in (load(300, 1), load(20000, 2), load(300, 3),
                   lambda s: s.seed(0, 0, 9000, slpic.SEED_GAP, e_lo=1.0, e_hi=50.0),
                   lambda s: s.clear_error(),
                   lambda s: s.set_launch_shape(8, 2),
                   load(1, 4)):
        for s in (sim, plain):
            change(s)
        with torch.cuda.stream(stream):
            graph.replay()
        plain.step(1)
        same(sim, plain)
    sim.close()
    plain.close()


@pytest.mark.parametrize("own", [False, True])
@pytest.mark.parametrize("call", ["count", "load", "seed"])
def test_change_of_stream_right_after_steps(slpic, call, own):  # noqa: F811
    """Calls on a new stream find the steps of the old one (the NULL stream, or
    one that does not wait for it) finished."""
    import torch
    spec = inputs.gap_spec(n_cells=64, V=300.0, pd_torr_cm=5.0, gamma_se=0.3, field_mode=1,
                           charge_shift=24)
    plain = make(slpic, 1)
    plain.step(40)
    plain.synchronize()
    old = torch.cuda.Stream() if own else torch.cuda.default_stream()
    sim = make(slpic, 1, old)
    torch.cuda.synchronize()
    with torch.cuda.stream(old):
        torch.cuda._sleep(20_000_000)  # about 10 ms: the steps start after the calls below
    sim.step(40)
    sim.set_stream(torch.cuda.Stream())
    for s in (sim, plain):
        if call == "load":
            for sp, m in enumerate(mixed_state(spec, 500, 200, seed=9)):
                s.load(0, sp, m)
        elif call == "seed":
            s.seed(0, 0, 700, slpic.SEED_GAP, e_lo=1.0, e_hi=50.0)
        else:
            s.count(0, 0)
        if call != "count":
            s.step(3)
    same(sim, plain)
    sim.close()
    plain.close()


@pytest.mark.parametrize("call", ["count", "field", "charge", "history", "seed"])
def test_replays_on_the_null_stream(slpic, call):  # noqa: F811
    """A call on a stream that does not wait for the NULL stream finds the
    steps replayed there finished."""
    import torch
    field_mode = 0 if call == "charge" else 1
    stream = torch.cuda.Stream()
    sim, plain = make(slpic, field_mode, stream), make(slpic, field_mode)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        sim.step(2)
    plain.step(4)
    plain.synchronize()
    args = {"field": (0,), "history": (0,),
            "seed": (0, 0, 700, slpic.SEED_GAP, 1.0, 1.0, 50.0)}.get(call, (0, 0))
    want = getattr(plain, call)(*args)
    torch.cuda._sleep(20_000_000)
    graph.replay()
    graph.replay()
    got = getattr(sim, call)(*args)
    assert np.array_equal(np.asarray(got), np.asarray(want))
    same(sim, plain)
    sim.close()
    plain.close()


def test_device_arrays_filled_on_the_null_stream(slpic):  # noqa: F811
    """load_device on a stream that does not wait for the NULL stream takes the
    values that work queued there writes."""
    import torch
    sim, plain = make(slpic, 0, torch.cuda.Stream()), make(slpic, 0)
    m = sim.particles(0, 0)
    host = {k: torch.from_numpy(v.view(np.int32) if k == "id" else v).pin_memory()
            for k, v in m.items()}
    dev = {k: torch.zeros_like(v, device="cuda") for k, v in host.items()}
    sim.count(0, 0)
    torch.cuda.synchronize()
    torch.cuda._sleep(20_000_000)
    for k in dev:
        dev[k].copy_(host[k], non_blocking=True)
    sim.load_device(0, 0, dev, next_id=len(m["id"]))
    plain.load(0, 0, m, next_id=len(m["id"]))
    for s in (sim, plain):
        s.step(2)
    same(sim, plain)
    sim.close()
    plain.close()
