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
    pairs, the elastic scattering and beta on 2^28 draws
    (tests/rounding_check.cu)."""
    from paper_2103_12194_gb300 import build
    exe = str(tmp_path / "rounding_check")
    subprocess.check_call([build.nvcc()] + build.common_flags() +
                          ["-I", build.CSRC, os.path.join(HERE, "rounding_check.cu"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.split()[:5] == ["0"] * 5, out.stdout


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


def deposit_of(m, spec, vlim):
    """The fixed-point deposit of FP32 markers, as every step forms it."""
    f = np.float32
    v2 = m["vx"] * m["vx"] + m["vy"] * m["vy"] + m["vz"] * m["vz"]
    with np.errstate(divide="ignore"):
        beta = np.minimum(f(1), f(vlim) / np.sqrt(v2)) if math.isfinite(vlim) else f(1)
    q = np.rint((beta * m["wj"]) * f(2.0 ** spec["charge_shift"])).astype(np.int64)
    right = (q * (m["off"] * f(2.0 ** 24)).astype(np.int64)) >> 24
    out = np.zeros(spec["n_cells"] + 1, np.int64)
    np.add.at(out, m["cell"], q - right)
    np.add.at(out, m["cell"] + 1, right)
    return out


@pytest.mark.parametrize("field_mode", [0, 1])
@pytest.mark.parametrize("populations", [
    [(40_000, 20_000)],                                        # one gap
    [(0, 3000), (1, 0), (130, 1), (0, 0), (9000, 4000)],        # uneven ones: several per CTA
    [(k * 37 + 1, 300) for k in range(60)],                    # more gaps than CTAs take singly
])
def test_collision_items_and_births(slpic, oracle_mod, populations, field_mode):  # noqa: F811
    """One dense step of every process with emission: the births of each gap
    in the order of their parents, with their serial numbers, whatever items
    and CTAs they fall to, and the deposit of exactly the markers there are."""
    sim = slpic.Simulation(len(populations))
    specs, states = [], []
    for k, (ne, ni) in enumerate(populations):
        spec = inputs.gap_spec(n_cells=(64, 300, 1500)[k % 3], V=300.0, pd_torr_cm=20.0,
                               gamma_se=0.5, field_mode=field_mode, charge_shift=24, seed=7 + k,
                               instance=k)
        specs.append(spec)
        states.append(mixed_state(spec, ne, ni, seed=300 + k))
        sim.configure(k, spec, capacity=(2 * ne + ni + 256, ne + ni + 256))
    for k, (e, i) in enumerate(states):
        sim.load(k, 0, e)
        sim.load(k, 1, i)
    sim.step(1)
    born = emitted = 0
    for k, spec in enumerate(specs):
        ref = oracle_mod.Oracle(spec, precision=32)
        ref.load(0, states[k][0])
        ref.load(1, states[k][1])
        ref.step(1)
        h, g = ref.history()[-1], sim.history(k)[-1]
        for key in ("n_live", "n_coll", "n_abs", "n_see", "n_candidates"):
            assert np.array_equal(h[key], g[key]), (k, key)
        born += int(h["n_coll"][2])
        emitted += int(h["n_see"])
        for s, vlim in ((0, spec["vlim_e"]), (1, spec["vlim_i"])):
            m, r = sim.particles(k, s), ref.particles(s)
            assert np.array_equal(m["id"], r["id"].astype(np.uint32)), (k, s)
            assert np.array_equal(m["cell"], r["cell"]) and np.array_equal(
                m["off"], r["off"].astype(np.float32)), (k, s)
            assert np.array_equal(sim.charge(k, s), deposit_of(m, spec, vlim)), (k, s)
    assert born > 0 and emitted > 0
    sim.close()
