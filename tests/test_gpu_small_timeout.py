"""A grid barrier of the single-CTA path that runs out while other instances are
inside a step: every CTA leaves its step loop as one, so each store is left as
it was after a whole step."""
import numpy as np
import pytest

from .test_gpu_small import SHAPES, items_for, load, slpic  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("field_mode", [0, 1])
def test_stores_are_whole_after_a_time_out(slpic, field_mode):  # noqa: F811
    items = items_for(SHAPES, field_mode=field_mode)
    sim = load(slpic, items)
    # a limit that the slowest instance's step may exceed, so that the word is
    # set while some CTAs are still in the step before
    sim.set_spin_limit(50)
    for inst, barrier in ((3, 2), (0, 3), (2, 5)):
        sim.test_skip_barrier(inst, barrier)
        with pytest.raises(slpic.SlpicError) as e:
            sim.step_small(10)
        assert e.value.code == slpic.ERR_TIMEOUT
        sim.clear_error()
        for i, (spec, _, _) in enumerate(items):
            steps = len(sim.history(i))
            for s in (0, 1):
                p = sim.particles(i, s)
                if steps:
                    assert len(p["id"]) == sim.tallies(i)["n_live"][s], (i, s)
                assert np.all((p["cell"] >= 0) & (p["cell"] < spec["n_cells"])), (i, s)
                assert len(np.unique(p["id"])) == len(p["id"]), (i, s)
    sim.close()
