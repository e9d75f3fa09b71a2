"""The calls that a user of this framework makes, as cases to be measured.

A case is a mapping of plain values; its "kind" is one of

* "gap": one gap, started, advanced by ``steps`` steps and read out.  "start"
  is "cathode" or "gap" (seeded on the device, as in the README) or "load"
  (markers of both species that the program already holds);
* "batch": many uneven gaps of a Paschen curve in one context, as ``bench.py
  --batch`` runs them;
* "search": one batched breakdown search (``paschen_bisect``);
* "trend": the paper's own breakdown test, the ion-population trend of an
  avalanche from 100 electrons at rest (``ion_trend``).

A pass starts from the same state every time (field, counters and markers are
set anew), so it can be repeated, and its outputs are what such a program
reads: deposit, density, field, tallies, and the markers themselves where the
population is small enough for them to be read as a matter of course.
"""
import math

import numpy as np
import torch

from paper_2103_12194_gb300 import inputs, slpic

FIELDS = ("cell", "off", "vx", "vy", "vz", "wj", "id")
READ_MARKERS = 100_000   # a run starting from at most so many also returns its markers
L2_BYTES = 129_000_000


def listed():
    return [
        # the paper's breakdown run at 1 Torr cm (219 cells, five processes,
        # energy-dependent yield): a few hundred markers, latency only
        _trend("paper_trend_219", pd=1.0, cells=219, V=171.5, steps=146, windows=6),
        # one step on markers of both species, read back whole: the smallest
        # call of a program that drives the steps itself
        _gap("one_step_25k", start="load", n_e=20_000, n_i=5_000, cells=256, pd=1.0, V=300.0,
             steps=1, gamma=0.5),
        # the plain small case: 2e4 electrons at 1 eV at the cathode
        _gap("cathode_256", start="cathode", n_e=20_000, cells=256, pd=1.0, V=300.0, steps=160),
        # the same gap on the double-precision marker path, more electrons
        _gap("cathode_256_fp64", start="cathode", n_e=60_011, cells=256, pd=1.0, V=300.0,
             steps=40, bits=64),
        # a quasi-neutral plasma, standard PIC (no speed limit), both species
        # and the field's feedback
        _gap("plasma_pic", start="load", n_e=2_000_003, n_i=4_000_001, cells=1310, pd=6.0,
             V=262.0, steps=48, limit=0.0, weight=1.5e6, shift=16),
        # the single Paschen point: 1e6 electrons at the cathode, 4096 cells
        _gap("paschen_point", start="cathode", n_e=1_000_000, cells=4096, pd=1.0, V=300.0,
             steps=64),
        # the microbenchmark gap at full size: every electron speed-limited
        # (v_lim 1/8 of the median speed), self-consistent field
        _gap("micro_32m", start="gap", n_e=32_000_000, cells=4096, pd=1.0, V=300.0, steps=16,
             limit=4.133),
        # the same gap with the field imposed, as the paper holds it
        _gap("micro_8m_imposed", start="gap", n_e=8_000_000, cells=4096, pd=1.0, V=300.0,
             steps=32, limit=4.133, poisson=False),
        # collision-dense: a quarter of the electrons are candidates per step
        _gap("dense_4m", start="gap", n_e=4_000_000, cells=6339, pd=33.3, V=1430.0, steps=32),
        # the 100 Torr row of the paper's table: a grid beyond shared memory,
        # five processes, energy-dependent yield
        _gap("grid_21832", start="gap", n_e=1_300_000, cells=21832, pd=100.0, V=1400.0,
             steps=32, limit=1.0, levels=3, energy_yield=True),
        # 32 uneven gaps of a Paschen curve in the same launches
        {"name": "batch_32", "kind": "batch", "instances": 32, "n_lo": 2_500, "n_hi": 1_000_000,
         "pd_lo": 0.1, "pd_hi": 100.0, "max_cells": 16384, "steps": 48},
        # one round of the batched breakdown search, 7 voltages at 2 pressures
        {"name": "search_2x7", "kind": "search", "pd_lo": 0.5, "pd_hi": 1.0, "n_pd": 2, "n_v": 7,
         "rounds": 1, "n_seed": 1000, "V_lo": 100.0, "V_hi": 500.0},
    ]


def _gap(name, *, start, n_e, n_i=0, cells, pd, V, steps, limit=4.0, poisson=True, bits=32,
         gamma=0.07, levels=1, energy_yield=False, weight=1.0, shift=32):
    """limit: the electrons' speed limit in units of v0 = sqrt(2 e V / M); 0
    is standard PIC."""
    return {"name": name, "kind": "gap", "start": start, "n_e": n_e, "n_i": n_i, "cells": cells,
            "pd": pd, "V": V, "steps": steps, "limit": limit, "poisson": poisson, "bits": bits,
            "gamma": gamma, "levels": levels, "energy_yield": energy_yield, "weight": weight,
            "shift": shift}


def _trend(name, *, pd, cells, V, steps, windows):
    return {"name": name, "kind": "trend", "pd": pd, "cells": cells, "V": V, "steps": steps,
            "windows": windows}


def _log(rng, lo, hi):
    return lo * math.exp(rng.random() * math.log(hi / lo))


def _paschen_V(pd):
    """Paschen's law (A = 11.5, B = 176, gamma = 0.07) on its right branch."""
    return 176.0 * pd / (math.log(11.5 * pd) - math.log(math.log(1.0 + 1.0 / 0.07)))


def draw(rng):
    kind = rng.choice(("trend", "load", "load", "cathode", "cathode", "gap", "gap", "gap",
                       "batch", "search"))
    if kind == "trend":
        pd = _log(rng, 0.6, 4.0)
        # around this gas's own breakdown voltage
        case = _trend("", pd=pd, cells=round(218.3 * pd), V=rng.uniform(0.9, 1.1) *
                      (171.5 if pd < 1.2 else 171.5 * (pd / 1.2) ** 0.3),
                      steps=rng.randint(60, 200), windows=rng.randint(3, 6))
    elif kind == "batch":
        k = rng.randint(3, 40)
        case = {"kind": "batch", "instances": k, "n_lo": round(_log(rng, 700, 5_000)),
                "n_hi": round(_log(rng, 5e4, 1e6)), "pd_lo": _log(rng, 0.1, 0.5),
                "pd_hi": _log(rng, 10.0, 100.0), "max_cells": rng.choice((2048, 8191, 16384)),
                "steps": rng.randint(10, 48)}
    elif kind == "search":
        lo = _log(rng, 0.3, 0.5)
        case = {"kind": "search", "pd_lo": lo, "pd_hi": 2.0 * lo, "n_pd": rng.randint(1, 2),
                "n_v": rng.choice((3, 5, 7)), "rounds": 1, "n_seed": round(_log(rng, 200, 1000)),
                "V_lo": 100.0, "V_hi": rng.uniform(400.0, 500.0)}
    else:
        bits = 64 if rng.random() < 0.2 else 32
        top = {"load": 4e6, "cathode": 1e6, "gap": 2e7}[kind] * (1 if bits == 32 else 0.02)
        n = round(_log(rng, 3e3, top))
        pd = _log(rng, 0.6, 40.0)
        # markers x steps of at most a fifth of the largest listed case
        steps = max(1, min(rng.randint(1, 100), int(1e8 if bits == 32 else 3e6) // n))
        plasma = kind == "load"
        case = _gap("", start=kind, n_e=n, n_i=round(n * rng.uniform(0.2, 2.0)) if plasma else 0,
                    # at most one collision per step: dx up to lambda_min
                    cells=round(_log(rng, max(64, _lambda_cells(pd, 10 ** 9) // 4), 22000)), pd=pd,
                    V=max(170.0, rng.uniform(0.9, 1.4) * _paschen_V(max(pd, 1.0))), steps=steps,
                    limit=rng.choice((0.0, 1.0, 4.0, 4.0, 16.0)), poisson=rng.random() < 0.7,
                    bits=bits, levels=rng.choice((1, 1, 3)),
                    energy_yield=rng.random() < 0.3,
                    weight=1.5e6 if plasma else 1.0, shift=16 if plasma else 32)
    case.pop("name", None)
    return case


# ---------------------------------------------------------------------------
# What a program has in hand before the call
# ---------------------------------------------------------------------------

def _spec(case, seed, instance=0):
    V, cells = case["V"], case["cells"]
    v0 = inputs.ion_speed(V)
    limit = case.get("limit", 1.0)
    if limit:
        vlim, dt = limit * v0, 0.01 / cells / (limit * v0)
    else:
        vlim, dt = math.inf, 0.01 / cells / math.sqrt(2.0 * inputs.QE * V / inputs.ME)
    spec = inputs.gap_spec(n_cells=cells, V=V, pd_torr_cm=case["pd"], dt=dt, vlim_e=vlim,
                           gamma_se=case.get("gamma", 0.07),
                           field_mode=1 if case.get("poisson") else 0,
                           charge_shift=case.get("shift", 32), seed=seed, instance=instance,
                           table=inputs.make_table(levels=case.get("levels", 1)))
    spec["emission_model"] = 1 if case.get("energy_yield") else 0
    return spec


def _markers(n, cells, mass, e_lo, e_hi, weight, gen, bits):
    """n markers uniform over the gap, energies log-uniform in [e_lo, e_hi]
    eV, isotropic; on the GPU."""
    real = torch.float64 if bits == 64 else torch.float32

    def u():
        return torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)

    v = torch.sqrt(2.0 * inputs.QE / mass * e_lo * torch.exp(u() * math.log(e_hi / e_lo)))
    ct = 1.0 - 2.0 * u()
    st, ph = torch.sqrt(1.0 - ct * ct), 2.0 * math.pi * u()
    below_one = 1.0 - (2.0 ** -53 if bits == 64 else 2.0 ** -24)
    return {
        "cell": torch.randint(cells, (n,), generator=gen, device="cuda", dtype=torch.int32),
        "off": u().to(real).clamp(max=below_one),
        "vx": (v * ct).to(real), "vy": (v * st * torch.cos(ph)).to(real),
        "vz": (v * st * torch.sin(ph)).to(real),
        "wj": torch.full((n,), weight, device="cuda", dtype=real),
        "id": torch.arange(n, device="cuda", dtype=torch.int32),
    }


def _load_state(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return [_markers(case["n_e"], case["cells"], inputs.ME, 0.1, 200.0, case["weight"], gen,
                     case["bits"]),
            _markers(case["n_i"], case["cells"], inputs.M_AR, 0.01, 30.0, case["weight"], gen,
                     case["bits"])]


def _host(markers):
    out = {k: t.cpu().numpy() for k, t in markers.items()}
    out["id"] = out["id"].astype(np.uint32)
    return out


def _lambda_cells(pd, most):
    """Cells of dx = lambda_min / 4 in a 1 cm gap, clamped to 128 .. most."""
    t = inputs.make_table()
    smax = float(np.max(t["sig_el"].astype(np.float64) + t["sig_ex"] + t["sig_io"]))
    n_g = pd * inputs.TORR / (inputs.KB * 300.0)
    return int(min(most, max(128, math.ceil(4 * 0.01 * n_g * smax))))


def _spread(case, k, n, key):
    """Value k of n spread over [key_lo, key_hi] by equal ratios."""
    lo, hi = case[key + "_lo"], case[key + "_hi"]
    return lo * (hi / lo) ** (k / (n - 1) if n > 1 else 0.0)


def _batch(case, seed):
    out = []
    for k in range(case["instances"]):
        pd = _spread(case, k, case["instances"], "pd")
        spec = _spec({"pd": pd, "V": _paschen_V(pd) if pd > 0.3 else 1000.0, "limit": 4.0,
                      "poisson": True, "cells": _lambda_cells(pd, case["max_cells"])},
                     1000 * seed + k, k)
        out.append((spec, round(_spread(case, k, case["instances"], "n"))))
    return out


def _search(case, seed):
    out = []
    for p in range(case["n_pd"]):
        pd = _spread(case, p, case["n_pd"], "pd")
        for j in range(case["n_v"]):
            out.append(_spec({"pd": pd, "V": 300.0, "limit": 4.0,
                              "cells": _lambda_cells(pd, 16384)},
                             1000 * seed + len(out), len(out)))
    return out


def _capacity(case):
    """Markers of each species a gap has room for: short runs of large
    populations grow little, long ones of small populations many times; in
    one step the electrons at most double and gain one per ion."""
    n = case["n_e"] + case["n_i"]
    if case["steps"] == 1:
        return 2 * n + 1024
    return n + n // 4 + 65536 if n >= 10_000_000 else 8 * n + (1 << 17)


def prepare(case, seed):
    state = dict(case=case)
    if case["kind"] == "batch":
        state["gaps"] = gaps = _batch(case, seed)
        specs = [s for s, _ in gaps]
        caps = [(4 * n + 65536, 4 * n + 65536) for _, n in gaps]
    elif case["kind"] == "search":
        specs = _search(case, seed)
        caps = [(32 * case["n_seed"], 32 * case["n_seed"])] * len(specs)
    elif case["kind"] == "trend":
        specs = [_spec({**case, "levels": 3, "energy_yield": True}, seed)]
        caps = [(1 << 18, 1 << 18)]
    else:
        specs = [_spec(case, seed)]
        caps = [(_capacity(case), _capacity(case))]
        if case["start"] == "load":
            e, i = _load_state(case, seed)
            # the double-precision path takes markers from host memory
            state["markers"] = (e, i) if case["bits"] == 32 else (_host(e), _host(i))
    sim = slpic.Simulation(len(specs), stream=torch.cuda.current_stream(),
                           precision=case.get("bits", 32))
    for k, (spec, cap) in enumerate(zip(specs, caps)):
        sim.configure(k, spec, capacity=cap)
    sim.launch_shape()   # completes the configuration: the device memory is there
    # the marker slots of a gap whose markers are read out
    read = case["kind"] == "trend" or (
        case["kind"] == "gap" and case["n_e"] + case["n_i"] <= READ_MARKERS)
    state.update(sim=sim, specs=specs, slots=caps[0][0] if read else 0)
    return state


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def _empty(bits):
    real = np.float64 if bits == 64 else np.float32
    return {k: np.empty(0, slpic.DTYPES.get(k, real)) for k in FIELDS}


def _restart(state):
    """The vacuum field, no markers, counters at zero."""
    sim, none = state["sim"], _empty(state["case"].get("bits", 32))
    for k, spec in enumerate(state["specs"]):
        sim.set_voltage(k, spec["V"])
        sim.load(k, slpic.ELECTRON, none)
        sim.load(k, slpic.ION, none)
        sim.reset_counters(k)


def _tallies(sim, n):
    t = np.stack([sim.tallies(k) for k in range(n)])
    return {name: np.ascontiguousarray(t[name]) for name in t.dtype.names}


def _padded(markers, slots):
    """Marker arrays at one length whatever their number: the rest is zero."""
    out = {k: np.zeros(slots, np.int64 if k == "id" else a.dtype) for k, a in markers.items()}
    for k, a in markers.items():
        out[k][: a.size] = a
    return out


def _read(sim, n, slots):
    """What a program reads of n gaps; of a single one also the density and,
    with slots, its markers."""
    out = {"tallies": _tallies(sim, n)}
    for sp, name in ((slpic.ELECTRON, "electron"), (slpic.ION, "ion")):
        out[name + "_charge"] = np.concatenate([sim.charge(k, sp) for k in range(n)])
        if n == 1:
            out[name + "_density"] = sim.density(0, sp)
        if slots:
            out[name] = _padded(sim.particles(0, sp), slots)
    fields = [sim.field(k) for k in range(n)]
    out["phi"] = np.concatenate([f[0] for f in fields])
    out["E"] = np.concatenate([f[1] for f in fields])
    return out


def run(state):
    case, sim = state["case"], state["sim"]
    if case["kind"] == "search":
        for k, spec in enumerate(state["specs"]):
            sim.set_seed(k, spec["seed"])
        lo, hi, gain = sim.paschen_bisect([case["V_lo"]] * case["n_pd"],
                                          [case["V_hi"]] * case["n_pd"], n_v=case["n_v"],
                                          rounds=case["rounds"], n_seed=case["n_seed"])
        return {"Vb_lo": lo, "Vb_hi": hi, "gain": gain, "tallies": _tallies(sim, gain.size)}
    if case["kind"] == "trend":
        _restart(state)
        sim.seed(0, slpic.ELECTRON, 100, slpic.SEED_REST)
        means, above = sim.ion_trend(case["steps"], case["windows"])
        return {"means": means, "above": above, **_read(sim, 1, state["slots"])}
    if case["kind"] == "batch":
        _restart(state)
        for k, (_, n) in enumerate(state["gaps"]):
            sim.seed(k, slpic.ELECTRON, n, slpic.SEED_GAP, e_lo=0.1, e_hi=200.0)
        sim.step(case["steps"])
        return _read(sim, len(state["gaps"]), 0)
    if case["start"] == "load":
        sim.set_voltage(0, case["V"])
        sim.reset_counters(0)
        for sp, m in enumerate(state["markers"]):
            n = len(m["cell"])
            if case["bits"] == 32:
                sim.load_device(0, sp, m, n)
            else:
                sim.load(0, sp, m, n)
    else:
        _restart(state)
        if case["start"] == "cathode":
            sim.seed(0, slpic.ELECTRON, case["n_e"], slpic.SEED_CATHODE, e0=1.0)
        else:
            sim.seed(0, slpic.ELECTRON, case["n_e"], slpic.SEED_GAP, e_lo=0.1, e_hi=200.0)
    sim.step(case["steps"])
    return _read(sim, 1, state["slots"])


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: a marker's state (seven fields) is read and what a push changes
    of it (cell, offset, v_x) written, in every step while the population is
    larger than the L2 cache, once per pass where it fits, and the grids'
    outputs.  Operations: about 100 per marker-step (gather, the limited
    kick's roots, divisions and logarithms, drift, the collision draw, the
    deposit).  Populations are taken at their size at the start."""
    real = 8 if case.get("bits") == 64 else 4
    per_marker = (2 * 4 + 5 * real) + (4 + 2 * real)
    if case["kind"] == "trend":
        n, steps, nodes = 500, case["steps"] * case["windows"], case["cells"] + 1
    elif case["kind"] == "search":
        # an avalanche crosses the gap in about a step per cell
        cells = sum(_lambda_cells(_spread(case, p, case["n_pd"], "pd"), 16384)
                    for p in range(case["n_pd"]))
        n, steps, nodes = case["n_seed"] * case["n_pd"] * case["n_v"], cells // case["n_pd"], 0
    elif case["kind"] == "batch":
        k = case["instances"]
        n = sum(round(_spread(case, j, k, "n")) for j in range(k))
        steps = case["steps"]
        nodes = sum(_lambda_cells(_spread(case, j, k, "pd"), case["max_cells"]) + 1
                    for j in range(k))
    else:
        n, steps, nodes = case["n_e"] + case["n_i"], case["steps"], case["cells"] + 1
    trips = steps if n * per_marker > L2_BYTES else 1
    return {"bytes": float(n * per_marker * trips + nodes * 48), "flops": 100.0 * n * steps}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------

def exact(case, seed):
    """One step from loaded markers, in 64 bits.  Longer runs have no such
    value: a Monte-Carlo avalanche is a chain of comparisons (a draw below a
    rate, a position beyond a cell), and 64-bit arithmetic takes another one
    of them sooner or later; from there the two are different avalanches."""
    if case["kind"] != "gap" or case["start"] != "load" or case["steps"] != 1 or \
            case["n_e"] + case["n_i"] > READ_MARKERS:
        return None
    return _OneStep(case, seed).outputs()


def _philox4(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on arrays of counters."""
    m = np.uint64(0xFFFFFFFF)
    c = [np.broadcast_to(np.asarray(x, np.uint64), np.shape(c0)) for x in (c0, c1, c2, c3)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32 & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [p1 >> np.uint64(32) ^ c[1] ^ np.uint64(k0), p1 & m,
             p0 >> np.uint64(32) ^ c[3] ^ np.uint64(k1), p0 & m]
        k0, k1 = k0 + 0x9E3779B9 & 0xFFFFFFFF, k1 + 0xBB67AE85 & 0xFFFFFFFF
    return [_uniform(x) for x in c]


def _philox2(c0, key):
    """First word of Philox2x32-10 with counter (c0, 0), as a uniform."""
    m = np.uint64(0xFFFFFFFF)
    a, b = np.asarray(c0, np.uint64), np.zeros(np.shape(c0), np.uint64)
    for _ in range(10):
        p = np.uint64(0xD256D193) * a
        a, b = p >> np.uint64(32) ^ b ^ np.uint64(key), p & m
        key = key + 0x9E3779B9 & 0xFFFFFFFF
    return _uniform(a)


def _uniform(x):
    return ((x >> np.uint64(9)).astype(np.float64) + 0.5) * 2.0 ** -23


def _turn(u, cc, sc, cp, sp):
    """Unit vectors u turned by the polar angle (cc, sc) and the azimuth
    (cp, sp), about the x axis' frame, or the z axis' where |u_x| > 0.99."""
    x, y, z = u
    near = np.abs(x) > 0.99
    w = np.sqrt(1 - np.where(near, z, x) ** 2)
    a = (x * cc + sc * cp * w, y * cc + sc * (z * sp - x * y * cp) / w,
         z * cc - sc * (y * sp + x * z * cp) / w)
    b = (x * cc + sc * (y * sp - z * x * cp) / w, y * cc - sc * (x * sp + z * y * cp) / w,
         z * cc + sc * cp * w)
    return [np.where(near, q, p) for p, q in zip(a, b)]


def _isotropic(speed, ua, ub):
    ct = 1 - 2 * ua
    st, ph = np.sqrt(1 - ct * ct), 2 * math.pi * ub
    return [speed * ct, speed * st * np.cos(ph), speed * st * np.sin(ph)]


class _OneStep:
    """One step of the method from the vacuum field, on numpy arrays."""

    def __init__(self, case, seed):
        self.case, self.seed, self.s = case, seed, _spec(case, seed)
        self.dx = self.s["d"] / self.s["n_cells"]
        self.n_g = self.s["p_Pa"] / (inputs.KB * self.s["T_K"])
        self.lost = np.zeros((2, 2))
        self.w_see = 0.0
        marks = [{k: v.astype(np.float64 if k in FIELDS[1:6] else np.int64)
                  for k, v in _host(m).items()} for m in _load_state(case, seed)]
        self.next_id = [len(m["cell"]) for m in marks]
        kept, self.emitted = [], []
        for sp, m in enumerate(marks):
            kept.append(self._advance(sp, m))
        self._collide(*kept)

    def _kick(self, sp, m):
        """dv_x/dt = beta q E / m over the step with E held: along the force,
        the integral of max(L, |v|) dv_x grows by L |A|."""
        s = self.s
        q, mass, L = (s[k + "_" + "ei"[sp]] for k in ("charge", "mass", "vlim"))
        A = q / mass * s["dt"] * (-s["V"] / s["d"])
        vx = m["vx"]
        if not math.isfinite(L):
            return vx + A, np.ones_like(vx)
        g, p2 = math.copysign(1.0, A), m["vy"] ** 2 + m["vz"] ** 2
        edge, p = np.sqrt(np.maximum(L * L - p2, 0)), np.sqrt(p2)

        def cost(w):
            a = np.maximum(np.abs(w), edge)
            with np.errstate(divide="ignore", invalid="ignore"):
                d = 0.5 * (a * np.hypot(a, p) - edge * np.hypot(edge, p) +
                           np.where(p2 > 0, p2 * (np.arcsinh(a / p) - np.arcsinh(edge / p)), 0))
            return np.copysign(L * np.minimum(np.abs(w), edge) + d, w)

        lo, hi = g * vx, g * vx + abs(A)
        goal = cost(lo) + L * abs(A)
        for _ in range(70):
            mid = 0.5 * (lo + hi)
            over = cost(mid) > goal
            lo, hi = np.where(over, lo, mid), np.where(over, mid, hi)
        vx = g * 0.5 * (lo + hi)
        with np.errstate(divide="ignore"):
            return vx, np.minimum(1.0, L / np.sqrt(vx ** 2 + p2))

    def _advance(self, sp, m):
        s = self.s
        m["vx"], beta = self._kick(sp, m)
        x = m["off"] + beta * m["vx"] * s["dt"] / self.dx
        step = np.floor(x)
        m["cell"], m["off"] = m["cell"] + step.astype(np.int64), x - step
        out = [m["cell"] < 0, m["cell"] >= s["n_cells"]]
        self.lost[sp] = [m["wj"][o].sum() for o in out]
        if sp == 1:
            c = out[0]
            g = np.full(c.sum(), s["gamma_se"])
            if s["emission_model"]:
                e = 0.5 * s["mass_i"] / inputs.QE * sum(m[k][c] ** 2 for k in ("vx", "vy", "vz"))
                g = 0.09 * (e / 700) ** np.where(e < 700, 0.05, 0.72)
            emit = _philox4(m["id"][c], 0, 1, 0, self.seed)[0] < g
            self.emitted = m["wj"][c][emit]
            self.w_see = self.emitted.sum()
        live = ~(out[0] | out[1])
        return {k: v[live] for k, v in m.items()}

    def _collide(self, e, ions):
        s, kv = self.s, 2 * inputs.QE / inputs.ME
        n_exc = s["n_exc"]
        grid = inputs.table_grid(s["tab_lo_exp2"], s["tab_log2_sub"], s["tab_octaves"])
        names = ["sig_el", "sig_ex"] + ["sig_ex%d" % k for k in range(2, n_exc + 1)] + ["sig_io"]
        table = np.cumsum([s[k].astype(np.float64) for k in names], axis=0)
        top = min(s["vlim_e"], math.sqrt(grid[-1] * kv))
        P0 = self.n_g * s["dt"] * top * table[-1].max()
        key = (self.seed ^ self.seed >> 32) & 0xFFFFFFFF ^ 0x85EBCA6B
        c = np.flatnonzero(_philox2(e["id"], key) < P0)
        v = [e[k][c] for k in ("vx", "vy", "vz")]
        speed = np.sqrt(sum(x * x for x in v))
        eps = speed ** 2 / kv
        u = _philox4(e["id"][c], 0, 0, 0, self.seed)
        rate = self.n_g * s["dt"] * np.minimum(speed, top) * \
            np.array([np.interp(eps, grid, t) for t in table])
        proc = (u[1] * P0 >= rate).sum(axis=0)
        new = [x.copy() for x in v]

        def put(sel, value):
            for x, y in zip(new, value):
                x[sel] = y

        k = proc == 0
        ek, u2 = eps[k], u[2][k]
        omc = np.clip(2 * np.expm1(u2 * np.log1p(ek)) / ek, 0, 2)
        opc = np.clip(-2 * (1 + ek) * np.expm1((u2 - 1) * np.log1p(ek)) / ek, 0, 2)
        ph = 2 * math.pi * u[3][k]
        turned = _turn([x[k] / speed[k] for x in v], np.where(omc <= 1, 1 - omc, opc - 1),
                       np.sqrt(omc * opc), np.cos(ph), np.sin(ph))
        after = np.sqrt(ek * (1 - 2 * inputs.ME / inputs.M_AR * omc) * kv)
        put(k, [after * x for x in turned])
        for lev in range(1, n_exc + 1):
            k = proc == lev
            left = np.maximum(eps[k] - s["e_ex" if lev == 1 else "e_ex%d" % lev], 0)
            put(k, _isotropic(np.sqrt(left * kv), u[2][k], u[3][k]))
        k = proc == n_exc + 1
        par = c[k]
        r1, r2 = (_philox4(e["id"][par], 0, 0, b, self.seed) for b in (1, 2))
        left = np.maximum(eps[k] - s["e_io"], 0)
        put(k, _isotropic(np.sqrt((left - r1[0] * left) * kv), u[2][k], u[3][k]))
        for name, x in zip(("vx", "vy", "vz"), new):
            e[name][c] = x
        born_e = _isotropic(np.sqrt(r1[0] * left * kv), r1[1], r1[2])
        r = math.sqrt(inputs.KB * s["T_K"] / inputs.M_AR) * \
            np.sqrt(-2 * np.log([r2[0], r2[2]]))
        a = 2 * math.pi * np.array([r2[1], r2[3]])
        born_i = [r[0] * np.cos(a[0]), r[0] * np.sin(a[0]), r[1] * np.cos(a[1])]
        self.w_ionz = e["wj"][par].sum()
        z, w = np.zeros(len(self.emitted)), self.emitted
        zero = z.astype(np.int64)
        self.marks = []
        for sp, (m, born) in enumerate(((e, born_e), (ions, born_i))):
            add = {"cell": e["cell"][par], "off": e["off"][par], "vx": born[0], "vy": born[1],
                   "vz": born[2], "wj": e["wj"][par], "id": self.next_id[sp] + np.arange(len(par))}
            m = {f: np.concatenate([m[f], add[f]]) for f in FIELDS}
            if sp == 0:
                at = self.next_id[0] + len(par) + np.arange(len(w)) + 2 ** 31
                tail = {"cell": zero, "off": z, "vx": z, "vy": z, "vz": z, "wj": w, "id": at}
                m = {f: np.concatenate([m[f], tail[f]]) for f in FIELDS}
            self.marks.append(m)

    def _charge(self, sp):
        """Physical particles at the nodes, weighted linearly by beta w_j."""
        m, L = self.marks[sp], self.s["vlim_" + "ei"[sp]]
        with np.errstate(divide="ignore"):
            w = m["wj"] * np.minimum(1.0, L / np.sqrt(m["vx"] ** 2 + m["vy"] ** 2 + m["vz"] ** 2))
        n = self.s["n_cells"] + 1
        return np.bincount(m["cell"], w * (1 - m["off"]), n) + \
            np.bincount(m["cell"] + 1, w * m["off"], n)

    def _field(self, net):
        """phi and E on the nodes: phi'' = -rho / eps0 between 0 and V."""
        s, n, dx = self.s, self.s["n_cells"], self.dx
        if s["field_mode"] == 0:
            return s["V"] * np.arange(n + 1) / n, np.full(n + 1, -s["V"] / s["d"])
        C = inputs.QE * dx / (s["area"] * 8.8541878128e-12)
        drop = C * np.concatenate([[0.0], np.cumsum(net[1:n])])  # of phi's slope, cell by cell
        slope = (s["V"] + drop.sum()) / n - drop
        E = np.empty(n + 1)
        E[0], E[1:n], E[n] = -slope[0], -0.5 * (slope[:-1] + slope[1:]), -slope[-1]
        return np.concatenate([[0.0], np.cumsum(slope)]), E / dx

    def outputs(self):
        charge = [self._charge(0), self._charge(1)]
        vol = np.full(len(charge[0]), self.s["area"] * self.dx)
        vol[[0, -1]] *= 0.5
        phi, E = self._field(charge[1] - charge[0])
        t = {name: None for name in slpic.TALLY_DTYPE.names}
        t.update(w_live=np.array([[m["wj"].sum() for m in self.marks]]), w_abs=self.lost[None],
                 w_see=np.array([self.w_see]), w_ionz=np.array([self.w_ionz]),
                 w_cath_ion=np.array([self.lost[1, 0]]))
        out = {"tallies": t, "phi": phi, "E": E}
        for sp, name in enumerate(("electron", "ion")):
            slots = _capacity(self.case)
            out[name] = {f: v if f in FIELDS[1:6] else None
                         for f, v in _padded(self.marks[sp], slots).items()}
            out[name + "_charge"] = None
            out[name + "_density"] = charge[sp] / vol
        return out
