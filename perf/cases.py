"""Performance cases: the calls that users of this library make, from one step of a small
system to whole trajectories of millions of species.

Every case is a dict of plain values with a ``kind``:

* ``noalloc``  one FP64 step on the caller's own device buffers (``chem_step_noalloc``);
* ``uniform``  a homogeneous mixture advanced with a fixed time step;
* ``volume``   a homogeneous mixture of the volume-scaling study, log-growing time step;
* ``tracks``   one pulse of proton tracks from 1 ps on, log-growing time step;
* ``pulses``   several square pulses, species carried step by step between them;
* ``sweep``    many independent pulse trains in one batched context;
* ``hybrid``   trains that alternate the step-by-step stage and the rate equations;
* ``beam_off`` the rate-equation stage alone, many trains.

A pass of a context is what a program does per trajectory with a context that it keeps:
reset, inject from host arrays, advance, read the tallies and the final species.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2509_03313_gb300 import chem, hybrid, workloads as W

N_TYPES = len(W.SPECIES)
N_RXN = len(W.WATER_REACTIONS)
# species left at the end of a beam-on stage, per 1,150 (the counts of the beam-off case)
BEAM_OFF_MIX = (250, 300, 60, 320, 70, 60, 90)
# steps per graph replay, grid limit, search mapping chosen per step, one kernel per phase:
# what the autotuner picks on large single trains and on the sweep
TUNED_TRACKS = (8, 255, -1, chem.CHEM_LAUNCH_PHASES)
TUNED_SWEEP = (8, 128, -1, chem.CHEM_LAUNCH_PHASES)


def listed():
    return [
        # the smallest call: a host program steps its own 2,000 species once (test size)
        {"name": "noalloc_2000", "kind": "noalloc", "n": 2000, "L": 200.0, "dt": 1e-9},
        # the plain single pulse: 2,000 species in 1 um, 1,000 steps of 1 ns, FP64
        {"name": "uniform_2000_fp64", "kind": "uniform", "precision": "fp64", "n": 2000, "L": 1000.0,
         "dt": 1e-9, "steps": 1000},
        # its dense variant in 200 nm, FP32-local: short runs of a small study
        {"name": "dense_2000_fp32", "kind": "uniform", "precision": "fp32", "n": 2000, "L": 200.0,
         "dt": 1e-9, "steps": 200},
        # one box of the volume-scaling study: 31,250 species in 0.5 um
        {"name": "volume_500_fp32", "kind": "volume", "precision": "fp32", "L": 500.0, "t_end": 2e-6},
        # the CPU baseline's box: 32,000 track species in 1.6 um, FP64, an odd end time
        {"name": "tracks_32k_fp64", "kind": "tracks", "precision": "fp64", "L": 1600.0, "t_end": 0.83e-6,
         "tuned": False},
        # the headline workload: 200 tracks of 5,000 species in 5 um, 1 ps to 1 us
        {"name": "tracks_1e6_fp32", "kind": "tracks", "precision": "fp32", "L": 5000.0, "t_end": 1e-6,
         "tuned": True},
        # the same in FP64, default launch settings
        {"name": "tracks_1e6_fp64", "kind": "tracks", "precision": "fp64", "L": 5000.0, "t_end": 1e-6,
         "tuned": False},
        # beyond the L2: 4.1e6 species in 8 um
        {"name": "tracks_4e6_fp32", "kind": "tracks", "precision": "fp32", "L": 8000.0, "t_end": 1e-6,
         "tuned": True},
        # build-up over two 1 us pulses 0.1 ms apart, step by step throughout, every track an
        # arrival of its own (the multi-pulse run's density in a 2.5 um box)
        {"name": "pulses_2_fp32", "kind": "pulses", "pulses": 2, "tracks": 40, "per_track": 1800,
         "L": 2500.0, "period": 1e-4},
        # the dose-rate sweep: 64 trains of 1e4 to 2e6 species in one context, 10 us window
        {"name": "sweep_64_fp32", "kind": "sweep", "trains": 64, "scale": 1.0},
        # dose series: 1, 3 and 5 pulses at two dose rates, each followed by 10 s of beam-off
        {"name": "hybrid_6_fp32", "kind": "hybrid", "most_pulses": 5, "species": 20000},
        # the beam-off stage of a sweep alone: 64 trains, 10 s of rate equations
        {"name": "beam_off_64", "kind": "beam_off", "trains": 64, "n_min": 500, "n_max": 20000,
         "t_off": 10.0},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("noalloc", "uniform", "uniform", "volume", "tracks", "tracks", "tracks", "pulses", "sweep",
                       "hybrid", "beam_off"))
    prec = rng.choice(("fp32", "fp64"))
    if kind == "noalloc":
        n = int(_log(rng, 40, 16001))
        return {"kind": kind, "n": n, "L": round(rng.uniform(200.0, 1000.0) * max(1.0, (n / 2000) ** (1 / 3)), 1),
                "dt": float("%.3g" % _log(rng, 1e-12, 1e-9))}
    if kind == "uniform":
        n = int(_log(rng, 200, 60000))
        return {"kind": kind, "precision": prec, "n": n,
                "L": round(rng.uniform(200.0, 1000.0) * max(0.75, (n / 2000) ** (1 / 3)), 1), "dt": 1e-9,
                "steps": rng.randint(20, 400)}
    if kind == "volume":
        return {"kind": kind, "precision": prec, "L": round(_log(rng, 200.0, 1000.0), 1),
                "t_end": float("%.3g" % _log(rng, 2e-7, 3e-6))}
    if kind == "tracks":
        return {"kind": kind, "precision": prec,
                "L": round(_log(rng, 500.0, 8000.0 if prec == "fp32" else 5000.0), 1),
                "t_end": float("%.3g" % _log(rng, 1e-9, 1e-6)), "tuned": rng.random() < 0.5}
    if kind == "pulses":
        return {"kind": kind, "pulses": rng.randint(2, 3), "tracks": int(_log(rng, 4, 27)),
                "per_track": int(_log(rng, 200, 1800)), "L": round(rng.uniform(1500.0, 2500.0), 1),
                "period": float("%.3g" % _log(rng, 5e-6, 1e-4))}
    if kind == "sweep":
        return {"kind": kind, "trains": rng.randint(2, 64), "scale": float("%.3g" % _log(rng, 0.05, 1.0))}
    if kind == "hybrid":
        return {"kind": kind, "most_pulses": rng.randint(1, 4), "species": int(_log(rng, 1000, 20000))}
    return {"kind": kind, "trains": rng.randint(1, 64), "n_min": 300, "n_max": int(_log(rng, 400, 20000)),
            "t_off": float("%.3g" % _log(rng, 1e-6, 10.0))}


# ------------------------------------------------------------------------------ inputs
def _mixture(n, mix=W.MIX_COUNTS):
    """n species in the ratio of `mix` (the remainder goes to the first type)."""
    mix = np.asarray(mix, dtype=np.int64)
    counts = mix * n // mix.sum()
    counts[0] += n - counts.sum()
    return counts


def _workloads(case, seed):
    """(workloads, plans): one workload per train; plans only for the hybrid case."""
    kind = case["kind"]
    if kind in ("noalloc", "uniform"):
        pulse = W.uniform_mixture(_mixture(case["n"]), case["L"], seed, energy_eV=case["n"] * 100.0 / 6.0)
        dt = case["dt"]
        return [W.Workload("uniform", case["L"], [pulse], W.Schedule(dt, dt), t_end=case.get("steps", 1) * dt)], None
    if kind == "volume":
        return [W.volume_scaling(case["L"], seed, t_end=case["t_end"])], None
    if kind == "tracks":
        return [W.tracks_same_density(seed, case["L"], t_end=case["t_end"])], None
    if kind == "pulses":
        return [W.multi_pulse(seed, n_pulses=case["pulses"], period_s=case["period"], n_tracks=case["tracks"],
                              species_per_track=case["per_track"], L=case["L"])], None
    if kind == "sweep":
        return W.batched_sweep(case["trains"], seed, case["scale"]), None
    if kind == "hybrid":
        series = sorted({1, (1 + case["most_pulses"]) // 2, case["most_pulses"]})
        wls, plans, _ = W.dose_series(n_pulses=series, species_per_pulse=case["species"], seed=seed)
        return wls, plans
    sizes = np.logspace(math.log10(case["n_min"]), math.log10(case["n_max"]), case["trains"]).astype(int)
    out = []
    for b, n in enumerate(sizes):
        L = 5000.0 * (int(n) / 1e5) ** (1.0 / 3.0)
        pulse = W.uniform_mixture(_mixture(int(n), BEAM_OFF_MIX), L, seed + 7919 * b, energy_eV=n * 20.0)
        out.append(W.Workload("beam_off", L, [pulse], W.Schedule(1e-11, 1e-7, W.LOG_GROWTH_20_PER_DECADE),
                              t_end=case["t_off"]))
    return out, None


class _Context:
    """A library context, destroyed with the state that holds it."""

    def __init__(self, cfgs, keep):
        self.keep = keep
        self.ctx = chem.chem_init(cfgs[0]) if len(cfgs) == 1 else chem.chem_batch_init(cfgs)

    def __del__(self):
        ctx, self.ctx = getattr(self, "ctx", None), None
        if ctx:
            chem.chem_destroy(ctx)


def prepare(case, seed):
    kind = case["kind"]
    wls, plans = _workloads(case, seed)
    alloc = chem.torch_allocator(0)
    state = {"case": case, "seed": seed, "wls": wls, "plans": plans}
    if kind == "noalloc":
        wl, p = wls[0], wls[0].pulses[0]
        cfg, keep = chem.make_config(wl.L, wl.D, wl.reactions, seed=seed, dt_min=case["dt"], dt_max=case["dt"],
                                     stream=torch.cuda.current_stream().cuda_stream)
        dev, most = torch.device("cuda", 0), chem.CHEM_NOALLOC_MAX_SPECIES
        words = ctypes.sizeof(chem.chem_event) // 4
        state.update(
            cfg=cfg, keep=keep, n=p.n, ids=torch.arange(p.n, dtype=torch.int32, device=dev),
            types=torch.from_numpy(p.types).to(dev), xyz=torch.from_numpy(np.ascontiguousarray(p.xyz)).to(dev),
            id_out=torch.zeros(most, dtype=torch.int32, device=dev),
            type_out=torch.zeros(most, dtype=torch.int32, device=dev),
            xyz_out=torch.zeros((most, 3), dtype=torch.float64, device=dev),
            ev_out=torch.zeros((most // 2, words), dtype=torch.int32, device=dev),
            n_out=torch.zeros(3, dtype=torch.int32, device=dev))
        torch.cuda.synchronize()
        return state
    fp64 = case.get("precision") == "fp64"
    cfgs, keep = [], [alloc]
    for b, wl in enumerate(wls):
        s, n = wl.schedule, wl.n_species
        if kind == "hybrid":
            cap, cand, cells = int(n * 0.8) + 4096, max(4096, n // 4), 128
        elif kind == "sweep":
            cap, cand, cells = int(n * 1.3) + 4096, max(4096, n // 2), 0
        elif kind == "beam_off":
            cap, cand, cells = n + 4096, max(4096, n // 4), 64
        else:
            cap, cand, cells = max(4096, int(1.4 * n)), max(4096, (7 * n) // 10), 0
        cfg, k = chem.make_config(
            wl.L, wl.D, wl.reactions, seed=seed + b, train_id=b,
            precision=chem.CHEM_FP64 if fp64 else chem.CHEM_FP32_LOCAL, dt_min=s.dt_min, dt_max=s.dt_max,
            dt_growth=s.dt_growth, reset_on_release=s.reset_on_release, cutoff_c=s.cutoff_c,
            sbs_horizon=s.sbs_horizon, capacity_species=cap, capacity_pending=n + 16, capacity_candidates=cand,
            cells_per_axis_max=cells, stream=torch.cuda.current_stream().cuda_stream, allocator=alloc)
        cfgs.append(cfg)
        keep.append(k)
    state["context"] = _Context(cfgs, keep)
    if kind not in ("hybrid", "beam_off"):
        most = cfgs[0].capacity_species
        state.update(ids=np.zeros(most, np.int32), types=np.zeros(most, np.int32), xyz=np.zeros((most, 3)))
    if kind == "sweep":
        chem.chem_set_tuning(state["context"].ctx, *TUNED_SWEEP)
    elif case.get("tuned") or kind == "pulses":
        chem.chem_set_tuning(state["context"].ctx, *TUNED_TRACKS)
    torch.cuda.synchronize()
    return state


# -------------------------------------------------------------------------------- run
def _run_noalloc(s):
    n_out = s["n_out"].data_ptr()
    st = chem.chem_step_noalloc(s["cfg"], 0, 0.0, s["case"]["dt"], s["n"], s["n"], s["ids"].data_ptr(),
                                s["types"].data_ptr(), s["xyz"].data_ptr(), s["id_out"].data_ptr(),
                                s["type_out"].data_ptr(), s["xyz_out"].data_ptr(), n_out, n_out + 4,
                                s["ev_out"].data_ptr(), n_out + 8)
    if st != chem.CHEM_OK:
        raise chem.ChemError(st, "chem_step_noalloc")
    return {k: s[k] for k in ("id_out", "type_out", "xyz_out", "ev_out", "n_out")}


def _read_state(s, train=None):
    """The final species into the arrays that the program keeps for them, [0, n) of each (the
    C entry point itself: the Python wrapper makes new arrays for every call)."""
    n = np.zeros(1, np.int64)
    ids, types, xyz = s["ids"], s["types"], s["xyz"]
    at = [v.ctypes.data_as(ctypes.c_void_p) for v in (types, ids, xyz, n)]
    lib, ctx, cap = chem.lib(), s["context"].ctx, ids.size
    st = lib.chem_get_state(ctx, cap, *at) if train is None else lib.chem_batch_get_state(ctx, train, cap, *at)
    if st != chem.CHEM_OK:
        raise chem.ChemError(st, chem.chem_last_error(ctx))
    return ids, types, xyz, int(n[0])


def run(state):
    kind = state["case"]["kind"]
    if kind == "noalloc":
        return _run_noalloc(state)
    ctx, wls = state["context"].ctx, state["wls"]
    seeds = [state["seed"] + b for b in range(len(wls))]
    if kind not in ("sweep", "hybrid", "beam_off"):
        wl = wls[0]
        chem.chem_reset(ctx, seeds[0])
        for p in wl.pulses:
            chem.chem_inject_pulse(ctx, p.types, p.xyz, p.t_arrival, p.energy_eV)
        chem.chem_run_until(ctx, wl.t_end)
        tally = chem.chem_tally(ctx, N_TYPES, N_RXN)
        ids, types, xyz, n = _read_state(state)
        return {"tally": tally, "ids": ids, "types": types, "xyz": xyz, "n": n}
    chem.chem_batch_reset(ctx, seeds)
    for b, wl in enumerate(wls):
        for p in wl.pulses:
            chem.chem_batch_inject(ctx, b, p.types, p.xyz, p.t_arrival, p.energy_eV)
    if kind == "hybrid":
        r = hybrid.run_plans(ctx, state["plans"], N_TYPES, N_RXN)
        return {k: r[k] for k in ("counts", "events", "extents", "t", "species_steps")}
    ends = [wl.t_end for wl in wls]
    if kind == "sweep":
        chem.chem_batch_run_until(ctx, ends)
    else:
        chem.chem_batch_run_homogeneous(ctx, ends)
    tallies = [chem.chem_batch_tally(ctx, b, N_TYPES, N_RXN) for b in range(len(wls))]
    out = {"counts": np.stack([t["counts"] for t in tallies]), "events": np.stack([t["events"] for t in tallies]),
           "G": np.stack([t["G"] for t in tallies]), "t": np.array([t["t"] for t in tallies]),
           "species_steps": np.array([t["species_steps"] for t in tallies])}
    if kind == "sweep":
        # the species of the smallest train (the sweep's product is the G-values above)
        ids, types, xyz, n = _read_state(state, 0)
        o = np.argsort(ids[:n])  # idle trains keep no order
        ids[:n], types[:n], xyz[:n] = ids[o], types[o], xyz[o]
        out.update(ids=ids, types=types, xyz=xyz, n=n)
    else:
        out["extents"] = np.stack([chem.chem_batch_homogeneous_report(ctx, b, N_RXN)[0] for b in range(len(wls))])
    return out


# ------------------------------------------------------------------------------- work
def _log_steps(t_end, dt_min, dt_max, growth=W.LOG_GROWTH_20_PER_DECADE):
    t, dt, n = 0.0, dt_min, 0
    while t < t_end and n < 10_000_000:
        if dt >= dt_max:
            return n + max(1, math.ceil((t_end - t) / dt_max - 1e-6))
        t, dt, n = t + dt, min(dt * growth, dt_max), n + 1
    return n


def work(case):
    """Bytes: the injected species read once and the final species written once (a species:
    position, type and arrival, 36 bytes), plus one read and one write of the state that every
    step advances (FP32-local 16 bytes, FP64 28 bytes a species) wherever a run has several
    steps. Operations: about 60 a species and step (displacement, wrap, cell) and 10 a pair
    inside the cutoff, of which a species has about two."""
    kind = case["kind"]
    state = 28 if kind == "noalloc" or case.get("precision") == "fp64" else 16
    if kind == "noalloc":
        n, live, steps = case["n"], case["n"], 1
    elif kind == "uniform":
        n, live, steps = case["n"], 0.9 * case["n"], case["steps"]
    elif kind == "volume":
        n = 2000 * (case["L"] / 200.0) ** 3
        live, steps = 0.6 * n, _log_steps(case["t_end"], 1e-12, 1.5e-8)
    elif kind == "tracks":
        n = max(1, round(200 * (case["L"] / 5000.0) ** 2)) * round(case["L"])
        live, steps = 0.75 * n, _log_steps(case["t_end"], 1e-12, 1e-6)
    elif kind == "pulses":
        n = case["pulses"] * case["tracks"] * case["per_track"]
        steps = case["pulses"] * case["tracks"] * 29 + (case["pulses"] - 1) * case["period"] / 1e-6
        live = 0.3 * n
    elif kind == "sweep":
        n = 2.5e6 * case["scale"] * case["trains"] / 64
        live, steps = 0.15 * n, 1459
    elif kind == "hybrid":
        n = 2 * case["most_pulses"] * 1.8 * case["species"]
        live, steps = 0.3 * n / case["most_pulses"], 300 * case["most_pulses"]
    else:
        # about 300 integrator steps of 21 substeps with a 9 x 9 solve each, per train
        return {"bytes": 2.0 * case["trains"] * (N_TYPES + N_RXN) * 8,
                "flops": case["trains"] * 300.0 * (6 * 600 + 21 * 300)}
    return {"bytes": 36.0 * (n + live) + (2.0 * state * live * steps if steps > 1 else 0.0),
            "flops": 80.0 * live * steps}


# ------------------------------------------------- the same results in 64 bits (numpy)
def _philox(c, key):
    """Philox4x32-10 (Salmon et al., SC'11) on four arrays of 32-bit words."""
    low, s = np.uint64(0xFFFFFFFF), np.uint64(32)
    x0, x1, x2, x3 = np.broadcast_arrays(*(np.asarray(v, np.uint64) for v in c))
    k0, k1 = (np.uint64(v) for v in key)
    for r in range(10):
        a, b = x0 * np.uint64(0xD2511F53), x2 * np.uint64(0xCD9E8D57)
        x0, x1, x2, x3 = (b >> s) ^ x1 ^ k0, b & low, (a >> s) ^ x3 ^ k1, a & low
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & low, (k1 + np.uint64(0xBB67AE85)) & low
    return x0, x1, x2, x3


def _u53(hi, lo):
    return (((hi << np.uint64(32)) | lo) >> np.uint64(11)).astype(np.float64)


def _simulate(wl, seed, full, steps, cells):
    """`steps` steps of length `full` of one FP64 train whose species all arrive at t = 0, on a
    hash of at most `cells` cells per axis (negative: a hash that starts finer than that and
    moves to one a sixth coarser than needed; it fixes the order in which species are listed:
    by cell, then by the last order, this step's products last)."""
    L, p = wl.L, wl.pulses[0]
    key = (seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF)
    ids, types, pos = np.arange(p.n), p.types.astype(np.int64), p.xyz.copy()
    rx = wl.reactions
    pair = np.full((N_TYPES, N_TYPES), -1)
    for r, x in enumerate(rx):
        pair[x.a, x.b] = pair[x.b, x.a] = r
    DAB = np.array([wl.D[x.a] + wl.D[x.b] for x in rx])
    R = np.array([x.k_tab for x in rx]) * 1e24 / 6.02214076e23 / (4.0 * math.pi * DAB)
    cut = R + wl.schedule.cutoff_c * np.sqrt(2.0 * DAB * full)
    n_cells = max(3, min(abs(cells), int(L / (cut.max() * 1.0001))))
    if cells < 0:
        n_cells = max(3, 5 * n_cells // 6)
    next_id, species_steps, events, t = p.n, 0, np.zeros(len(rx), np.int64), 0.0
    shell = [(dx, dy, dz) for dz in (0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1) if (dz, dy, dx) >= (0, 0, 0)]
    for step in range(steps):
        # a context's last step is trimmed to land on its end time
        dt = wl.t_end - t if steps > 1 and step == steps - 1 else full
        t, species_steps = t + full, species_steps + ids.size
        a, b = _philox((ids, step, 0, 0), key), _philox((ids, step, 0, 1), key)
        r1 = np.sqrt(-2.0 * np.log((_u53(a[0], a[1]) + 1.0) * 2.0 ** -53))
        r2 = np.sqrt(-2.0 * np.log((_u53(b[0], b[1]) + 1.0) * 2.0 ** -53))
        t1, t2 = (2.0 * math.pi * (_u53(q[2], q[3]) * 2.0 ** -53) for q in (a, b))
        move = np.sqrt(2.0 * wl.D[types] * dt)[:, None] * np.stack([r1 * np.cos(t1), r1 * np.sin(t1), r2 * np.cos(t2)], 1)
        pos = pos + move
        pos = pos - np.floor((pos + 0.5 * L) / L) * L
        pos = np.where(pos >= 0.5 * L, pos - L, np.where(pos < -0.5 * L, pos + L, pos))
        cell = np.clip(np.floor((pos + 0.5 * L) * (n_cells / L)).astype(np.int64), 0, n_cells - 1)
        code = (cell[:, 2] * n_cells + cell[:, 1]) * n_cells + cell[:, 0]
        o = np.argsort(code, kind="stable")
        ids, types, pos, move, cell, code = ids[o], types[o], pos[o], move[o], cell[o], code[o]
        # every pair of species in one cell or in a cell and one of its 13 forward neighbours
        ii, jj = [], []
        for d in shell:
            c = (cell + d) % n_cells
            c = (c[:, 2] * n_cells + c[:, 1]) * n_cells + c[:, 0]
            lo, hi = np.searchsorted(code, c, "left"), np.searchsorted(code, c, "right")
            if d == (0, 0, 0):
                lo = np.arange(ids.size) + 1
            m = np.maximum(hi - lo, 0)
            i = np.repeat(np.arange(ids.size), m)
            ii.append(i)
            jj.append(np.arange(i.size) - np.repeat(np.cumsum(m) - m, m) + lo[i])
        i, j = np.concatenate(ii), np.concatenate(jj)
        k = pair[types[i], types[j]]
        i, j, k = i[k >= 0], j[k >= 0], k[k >= 0]
        i, j = np.where(ids[i] < ids[j], i, j), np.where(ids[i] < ids[j], j, i)
        sep = pos[j] - pos[i]
        sep = np.where(sep >= 0.5 * L, sep - L, np.where(sep < -0.5 * L, sep + L, sep))
        d2 = (sep * sep).sum(1)
        near = d2 < cut[k] ** 2
        i, j, k, sep, d2 = i[near], j[near], k[near], sep[near], d2[near]
        d1, d0 = np.sqrt(d2), np.sqrt(((sep - (move[j] - move[i])) ** 2).sum(1))
        with np.errstate(all="ignore"):
            w = DAB[k] * dt
            prob = np.exp(-(d0 - R[k]) * (d1 - R[k]) / w) * np.expm1(-R[k] * (d0 + d1 - R[k]) / w) / np.expm1(-d0 * d1 / w)
        u = _philox((ids[i], step, ids[j], 2), key)
        hit = np.flatnonzero((d1 <= R[k]) | (d0 <= R[k]) | (_u53(u[0], u[1]) * 2.0 ** -53 < prob))
        gone, done = np.zeros(ids.size, bool), []
        for c in hit[np.lexsort((ids[j[hit]], ids[i[hit]], d2[hit]))]:
            if not (gone[i[c]] or gone[j[c]]):
                gone[i[c]] = gone[j[c]] = True
                done.append(c)
        new_t, new_x = [], []
        for c in sorted(done, key=lambda c: ids[i[c]]):
            Da, Db = wl.D[types[i[c]]], wl.D[types[j[c]]]
            at = pos[i[c]] + Da / (Da + Db) * sep[c]
            at = at - np.floor((at + 0.5 * L) / L) * L
            events[k[c]] += 1
            new_t += rx[k[c]].products
            new_x += [at] * len(rx[k[c]].products)
        ids = np.concatenate([ids[~gone], next_id + np.arange(len(new_t))])
        next_id += len(new_t)
        types = np.concatenate([types[~gone], np.array(new_t, np.int64)])
        pos = np.concatenate([pos[~gone], np.array(new_x, np.float64).reshape(-1, 3)])
    return ids, types, pos, events, species_steps


def _extents(wl, t_off):
    """Reaction extents of the rate equations after t_off: Radau IIA of order 5 (Hairer and
    Wanner, Solving ODEs II, Sec. IV.8) on a geometric grid of times. `wl`: list of trains."""
    n0 = np.stack([np.bincount(w.pulses[0].types, minlength=N_TYPES) for w in wl]).astype(np.float64)
    rx, V = wl[0].reactions, np.array([w.L ** 3 * 1e-24 for w in wl])
    a, b = np.array([r.a for r in rx]), np.array([r.b for r in rx])
    kap = np.array([r.k_tab * (0.5 if r.a == r.b else 1.0) for r in rx])[None, :] / (6.02214076e23 * V[:, None])
    nu = np.zeros((N_TYPES, len(rx)))
    for r, x in enumerate(rx):
        nu[x.a, r] -= 1
        nu[x.b, r] -= 1
        for q in x.products:
            nu[q, r] += 1
    s6 = math.sqrt(6.0)
    A = np.array([[(88 - 7 * s6) / 360, (296 - 169 * s6) / 1800, (-2 + 3 * s6) / 225],
                  [(296 + 169 * s6) / 1800, (88 + 7 * s6) / 360, (-2 - 3 * s6) / 225],
                  [(16 - s6) / 36, (16 + s6) / 36, 1 / 9]])
    B, m = len(wl), len(rx)
    e, t, first = np.zeros((B, m)), 0.0, 1e-12
    while t < t_off:
        h = min(max(first, 0.025 * t), t_off - t)
        n = n0 + e @ nu.T
        J = kap[:, :, None] * (n[:, b, None] * nu[a][None] + n[:, a, None] * nu[b][None])
        M = np.eye(3 * m) - h * np.einsum("ij,bkl->bikjl", A, J).reshape(B, 3 * m, 3 * m)
        Z, inv = np.zeros((B, 3, m)), np.linalg.inv(M)
        for _ in range(6):
            n = n0[:, None] + (e[:, None] + Z) @ nu.T
            f = kap[:, None] * n[..., a] * n[..., b]
            g = h * np.einsum("ij,bjk->bik", A, f) - Z
            dz = (inv @ g.reshape(B, 3 * m, 1)).reshape(B, 3, m)
            Z += dz
            if np.abs(dz).max() < 1e-11:
                break
        e, t = e + Z[:, 2], t + h
    return e


def exact(case, seed):
    """Positions, G-values and clock of small FP64 runs and the extents of the beam-off stage.
    FP32-local runs draw other random numbers than FP64 ones: they have no such value."""
    kind = case["kind"]
    if kind == "beam_off":
        wls, _ = _workloads(case, seed)
        return {"counts": None, "events": None, "G": None, "t": np.full(len(wls), case["t_off"]),
                "species_steps": None, "extents": _extents(wls, case["t_off"])}
    small = case.get("n", 10 ** 9) * case.get("steps", 1) <= 2_100_000 and case.get("n", 0) <= 20_000
    if not small or case.get("precision") == "fp32":
        return None
    wl = _workloads(case, seed)[0][0]
    p = wl.pulses[0]
    steps = case.get("steps", 1)
    cells = -31 if kind == "noalloc" else int(np.cbrt(max(4096, int(1.4 * p.n)) * 16.0))
    ids, types, pos, events, species_steps = _simulate(wl, seed, case["dt"], steps, cells)
    if kind == "noalloc":
        out = np.zeros((chem.CHEM_NOALLOC_MAX_SPECIES, 3))
        out[:ids.size] = pos
        return {"id_out": None, "type_out": None, "xyz_out": out, "ev_out": None, "n_out": None}
    counts = np.bincount(types, minlength=N_TYPES)
    tally = {"counts": counts, "G": counts * 100.0 / p.energy_eV, "events": events, "t": wl.t_end,
             "species_steps": species_steps}
    out = np.zeros((max(4096, int(1.4 * p.n)), 3))
    out[:ids.size] = pos
    return {"tally": tally, "ids": None, "types": None, "xyz": out, "n": ids.size}
