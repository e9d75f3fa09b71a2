"""The particle kernel's tiles and its branch-free kick, where they can go
wrong: fills around the passes of a tile and around whole tiles, species with
and without a speed limit and a deposit (which decide what is copied of a
tile), kicks outside the range of the branch-free arithmetic, that arithmetic
itself, and markers that are read from device memory where they are.

The bars are those of the parity tests: bit-exact against the oracle's FP32
mirror, or against CUDA's IEEE operations.
"""
import math
import os
import subprocess

import numpy as np
import pytest

from paper_2103_12194_gb300 import inputs

from .test_gpu_parity import assert_same_markers, mixed_state, slpic  # noqa: F401

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("field_mode", [0, 1])
@pytest.mark.parametrize("vlim_e,vlim_i", [(2e5, math.inf), (math.inf, math.inf), (math.inf, 900.0)])
def test_fills_around_passes_and_tiles(slpic, oracle_mod, field_mode, vlim_e, vlim_i):  # noqa: F811
    """Three vacuum steps of gaps holding 1 .. 257 markers of each species,
    many of which leave through the electrodes (ions emitting)."""
    fills = [(1, 2), (2, 1), (63, 65), (64, 64), (65, 63), (127, 129), (128, 128), (129, 127),
             (257, 192)]
    sim = slpic.Simulation(len(fills))
    specs, states = [], []
    for k, (ne, ni) in enumerate(fills):
        spec = inputs.gap_spec(n_cells=32, V=200.0, pd_torr_cm=1.0, gamma_se=0.6,
                               field_mode=field_mode, vlim_e=vlim_e, vlim_i=vlim_i,
                               dt=0.01 / 32 / 2e5, seed=3 + k, instance=k, charge_shift=24)
        spec["p_Pa"] = 0.0
        specs.append(spec)
        states.append(mixed_state(spec, ne, ni, seed=50 + k))
        sim.configure(k, spec, capacity=(2048, 2048))
    for k, (e, i) in enumerate(states):
        sim.load(k, 0, e)
        sim.load(k, 1, i)
    sim.step(3)
    left = 0
    for k, spec in enumerate(specs):
        ref = oracle_mod.Oracle(spec, precision=32)
        ref.load(0, states[k][0])
        ref.load(1, states[k][1])
        ref.step(3)
        h = ref.history()
        for key in ("n_live", "n_abs", "n_see"):
            assert np.array_equal(sim.history(k)[key], h[key]), (k, key)
        left += int(np.sum(h["n_abs"]))
        for s in (0, 1):
            # an imposed field's deposit is formed when it is read
            assert np.array_equal(sim.charge(k, s), ref.charge(s)), (k, s)
            if field_mode == 0:
                assert_same_markers(sim.particles(k, s), ref.particles(s), 2e5,
                                    exact_values=True)
    assert left >= len(fills)  # the case has markers that leave: one per gap or more
    sim.close()


@pytest.mark.parametrize("vlim", [3e-4, 1e5, 2e9])
@pytest.mark.parametrize("kick", [2e-7, 3e-6, 3e5, 3e9])
def test_kicks_outside_the_branch_free_range(slpic, oracle_mod, vlim, kick):  # noqa: F811
    """Limits and kicks inside and outside the range of the branch-free
    arithmetic, with speeds from 1e-3 to 1e12 m/s mixed in every warp: one
    vacuum step, bit-exact against the FP32 mirror."""
    n, cells = 700, 64
    V = 100.0
    dt = kick / (inputs.QE * (V / 0.01) / inputs.ME)
    spec = inputs.gap_spec(n_cells=cells, V=V, pd_torr_cm=1.0, gamma_se=0.0, field_mode=0,
                           vlim_e=vlim, dt=dt, seed=1)
    spec["p_Pa"] = 0.0
    st = inputs.gap_state(n, spec, rng_seed=9)
    rng = np.random.default_rng(4)
    top = 1e12 if vlim > 1.0 else 1e3
    for k in ("vx", "vy", "vz"):
        s = 10.0 ** rng.uniform(-3, math.log10(top), n) * rng.choice((-1.0, 1.0), n)
        st[k] = s.astype(np.float32)
    st["vy"][::7] = 0.0
    st["vz"][::7] = 0.0
    sim = slpic.Simulation(1)
    sim.configure(0, spec, capacity=(4096, 4096))
    sim.load(0, 0, st)
    sim.step(1)
    ref = oracle_mod.Oracle(spec, precision=32)
    ref.load(0, st)
    ref.step(1)
    assert_same_markers(sim.particles(0, 0), ref.particles(0), vlim, exact_values=True)
    sim.close()


def test_branch_free_operations_equal_the_ieee_ones(slpic, tmp_path):  # noqa: F811
    """sqrt_mid and rcp_mid on every float of their range, div_mid on 2^32
    pairs (tests/rounding_check.cu)."""
    from paper_2103_12194_gb300 import build
    exe = str(tmp_path / "rounding_check")
    subprocess.check_call([build.nvcc()] + build.common_flags() +
                          ["-I", build.CSRC, os.path.join(HERE, "rounding_check.cu"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.split()[:3] == ["0", "0", "0"], out.stdout


@pytest.mark.parametrize("start", [0, 1, 3])
def test_markers_read_from_device_memory(slpic, start):  # noqa: F811
    """load_device of views that begin inside an allocation gives the markers
    that load gives, and what is read back is what was loaded."""
    import torch
    n = 1000
    spec, _ = inputs.small_gap_config()
    st = inputs.gap_state(n + 8, spec, rng_seed=2)
    view = {k: v[start:start + n] for k, v in st.items()}
    dev = {k: torch.from_numpy(v.view(np.int32) if k == "id" else v).cuda()[start:start + n]
           for k, v in st.items()}
    sim = slpic.Simulation(1)
    sim.configure(0, spec, capacity=(2048, 2048))
    sim.load_device(0, 0, dev, n + 8)
    got = sim.particles(0, 0)
    for k in got:
        assert np.array_equal(got[k], view[k]), k
    sim.close()
