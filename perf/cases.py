"""What the compiler's users have it do, as measurable cases.

Every case goes through the package's public entry points: a ``Driver`` that
compiles one circuit or a batch (inputs on the device or on the host, the
hyperedges left on the device or written into page-locked host arrays), the
autograd function over a compile, and a ``Server`` that compiles the cycles of
many patches as they arrive.  Circuits come from the package's generators; the
noise vector is drawn log-uniformly from [1e-4, 3e-3] by the seed.

``exact`` is an independent analysis in plain numpy: the circuit is walked
backward once with, per qubit, the XOR of random 128-bit keys of the detectors
and observables an X or a Z error would flip (XOR of keys = key of the XOR of
sets), so equal keys are equal masks.
"""
import math

import numpy as np
import torch

from paper_2604_16613_gb300 import circuits as C
from paper_2604_16613_gb300.dem import Bounds, DemFunction, DeviceCircuit, Driver
from paper_2604_16613_gb300.serve import Server


def listed():
    return [
        # the smallest call: one distance-3 memory, inputs and result on the device (latency and launches)
        {"name": "surface3", "kind": "surface", "d": 3, "rounds": 3, "level": "L2", "z_only": False, "io": "device",
         "slack": 1.0},
        # a control system's call: host arrays in, hyperedges out in page-locked host arrays, on a driver whose
        # buffers were sized for a larger circuit
        {"name": "surface5_host", "kind": "surface", "d": 5, "rounds": 5, "level": "L2", "z_only": False, "io": "host",
         "slack": 8.0},
        # ordinary sizes of the distance sweep
        {"name": "surface11", "kind": "surface", "d": 11, "rounds": 11, "level": "L2", "z_only": False,
         "io": "device", "slack": 1.0},
        {"name": "surface15_L1", "kind": "surface", "d": 15, "rounds": 15, "level": "L1", "z_only": False,
         "io": "device", "slack": 1.0},
        # the headline compile
        {"name": "surface25", "kind": "surface", "d": 25, "rounds": 25, "level": "L2", "z_only": False,
         "io": "device", "slack": 1.0},
        # the cheapest model of the same experiment: L0 with the Z-check detectors only
        {"name": "surface25_L0_z", "kind": "surface", "d": 25, "rounds": 25, "level": "L0", "z_only": True,
         "io": "device", "slack": 1.0},
        # the headline compile end to end: host arrays in, hyperedges out on the host
        {"name": "surface25_host", "kind": "surface", "d": 25, "rounds": 25, "level": "L2", "z_only": False,
         "io": "host", "slack": 1.0},
        # fitting noise: forward and adjoint of the [[144,12,12]] code (non-local checks, twelve observables)
        {"name": "bb12_grad", "kind": "bb_grad", "rounds": 12, "level": "L2"},
        # a long memory of few qubits: many layers, a long observable
        {"name": "repetition25x100", "kind": "repetition", "d": 25, "rounds": 100, "level": "L2"},
        # the branches of an adaptive circuit, one batch (the largest: 13 M mechanisms)
        {"name": "adaptive16", "kind": "adaptive", "n": 16, "d": 10, "lo": 10, "hi": 30, "level": "L2"},
        # many small uneven circuits in one host call (a parameter scan, a test bench)
        {"name": "small_batch", "kind": "small_batch", "n": 64, "lo": 3, "hi": 7, "level": "L2"},
        # serving: patches that each issue a request per cycle; registered steady-state cycles, and one adaptive
        # patch whose cycles are submitted as rows
        {"name": "serve", "kind": "serve", "surface": 9, "bb": 2, "adaptive": 1, "cycles": 6, "k": 1, "level": "L2"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["surface", "surface", "surface", "bb_grad", "repetition", "adaptive", "small_batch", "serve"])
    level = rng.choice(["L0", "L1", "L2", "L2"])
    if kind == "surface":
        # up to the headline's distance with up to 30 rounds, and (short) experiments on more qubits than that
        d = _log_int(rng, 3, 45)
        rounds = rng.randint(1, max(1, min(30, 20000 // (d * d))))
        return {"kind": kind, "d": d, "rounds": rounds, "level": level, "z_only": rng.random() < 0.25,
                "io": rng.choice(["device", "host"]), "slack": rng.choice([1.0, 1.5, 4.0])}
    if kind == "bb_grad":
        return {"kind": kind, "rounds": rng.randint(1, 14), "level": level}
    if kind == "repetition":
        return {"kind": kind, "d": _log_int(rng, 3, 40), "rounds": _log_int(rng, 2, 150), "level": level}
    if kind == "adaptive":
        lo = rng.randint(4, 12)
        return {"kind": kind, "n": rng.randint(1, 14), "d": rng.choice([4, 6, 8, 10]), "lo": lo,
                "hi": lo + rng.randint(0, 14), "level": level}
    if kind == "small_batch":
        return {"kind": kind, "n": _log_int(rng, 4, 96), "lo": 3, "hi": rng.randint(3, 9), "level": level}
    return {"kind": kind, "surface": rng.randint(1, 9), "bb": rng.randint(0, 2), "adaptive": rng.randint(0, 1),
            "cycles": rng.randint(3, 6), "k": rng.randint(1, 4), "level": level}


# -- circuits -------------------------------------------------------------------------------------------------------

_NM = C.NoiseModel.uniform(1e-3)


def _circuits(case):
    """The circuits of a compile case (for "serve" one per patch, with more cycles than the run submits)."""
    k = case["kind"]
    if k == "surface":
        return [C.rotated_surface_code_memory(case["d"], case["rounds"], _NM, z_detectors_only=case["z_only"])]
    if k == "bb_grad":
        return [C.bb_memory(case["rounds"], _NM, seed=3)]
    if k == "repetition":
        return [C.repetition_code_memory(case["d"], case["rounds"], _NM)]
    if k == "adaptive":
        return C.adaptive_branches(n=case["n"], d=case["d"], lo=case["lo"], hi=case["hi"], seed=4, noise=_NM)
    if k == "small_batch":
        span = case["hi"] - case["lo"] + 1
        return [C.rotated_surface_code_memory(case["lo"] + i % span, 2 + (i * 5) % 7, _NM) for i in range(case["n"])]
    out = []
    for i in range(case["surface"]):
        out.append((C.rotated_surface_code_memory(5 + 2 * (i % 11), case["cycles"] + 3, _NM), 1))
    if case["bb"]:
        bb = C.bb_memory(case["cycles"] + 3, _NM, seed=3)
        out += [(bb, 1)] * case["bb"]
    for i in range(case["adaptive"]):
        out.append((C.concatenated_adaptive_branch(10, case["cycles"] + 7, seed=40 + i, noise=_NM), 5))
    return out


def _noise(circuits, seed):
    return np.concatenate([C.log_uniform_noise(c.n_locations, seed=1000 * int(seed) + i)
                           for i, c in enumerate(circuits)]).astype(np.float32)


def _serve_blocks(case, seed):
    """Per patch: (circuit, horizon, the cycle blocks submitted in order, registered?).  A surface or BB patch
    repeats its steady-state cycle, so its noise repeats too."""
    out = []
    for i, (c, h) in enumerate(_circuits(case)):
        blocks = c.cycle_blocks()
        registered = h == 1
        if registered:
            blocks = [blocks[0], blocks[1]]
        else:
            blocks = blocks[:case["cycles"]]
        for t, b in enumerate(blocks):
            b["noise"] = C.log_uniform_noise(b["n_locations"], seed=100000 * int(seed) + 100 * i + t).astype(np.float32)
        out.append((c, h, blocks, registered))
    return out


# -- prepare and run ------------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind, level = case["kind"], case["level"]
    if kind == "serve":
        patches = _serve_blocks(case, seed)
        srv = Server.for_circuits([p[0] for p in patches], max_cycles_per_step=case["k"],
                                  max_horizon=max(p[1] for p in patches))
        return {"kind": kind, "srv": srv, "patches": patches, "cycles": case["cycles"], "k": case["k"], "level": level}
    circs = _circuits(case)
    noise = _noise(circs, seed)
    slack = case.get("slack", 1.0)
    bounds = Bounds.for_circuits(circs, slack=slack)
    drv = Driver(bounds)
    state = {"kind": kind, "drv": drv, "level": level, "io": case.get("io", "device")}
    if kind == "small_batch":
        state.update(io="host_in", circuits=circs, noise=noise)
    elif state["io"] == "host":
        dem = drv.compile(circs[0], noise, level)
        out = {"det_offsets": torch.empty(dem.n_edges + 1, dtype=torch.int32, pin_memory=True),
               "det_idx": torch.empty(max(dem.n_det_entries, 1), dtype=torch.int32, pin_memory=True),
               "obs_mask": torch.empty(max(dem.n_edges, 1), dtype=torch.int64, pin_memory=True),
               "prob": torch.empty(max(dem.n_edges, 1), dtype=torch.float32, pin_memory=True),
               "logodds": torch.empty(max(dem.n_edges, 1), dtype=torch.float32, pin_memory=True)}
        drv.set_host_output(out)
        state.update(circuits=circs[0], noise=noise, out=out)
    else:
        dcs = [DeviceCircuit(c) for c in circs]
        state.update(circuits=dcs if kind == "adaptive" else dcs[0],
                     noise=torch.tensor(noise, dtype=torch.float32, device="cuda"))
    if kind == "bb_grad":
        e = drv.compile(state["circuits"], state["noise"], level).n_edges
        g = torch.Generator().manual_seed(int(seed))
        state["g"] = (torch.randn(e, generator=g).cuda(), (1e-3 * torch.randn(e, generator=g)).cuda())
        state["noise"].requires_grad_(True)
    return state


def run(state):
    if state["kind"] == "serve":
        return _run_serve(state)
    drv, level = state["drv"], state["level"]
    if state["kind"] == "bb_grad":
        prob, logodds = DemFunction.apply(state["noise"], drv, state["circuits"], level)
        (grad,) = torch.autograd.grad([prob, logodds], [state["noise"]], list(state["g"]))
        return {"prob": prob, "logodds": logodds, "grad": grad}
    dem = drv.compile(state["circuits"], state["noise"], level)
    if state["io"] == "host":
        o, e, n = state["out"], dem.n_edges, dem.n_det_entries
        return {"det_offsets": o["det_offsets"][:e + 1], "det_idx": o["det_idx"][:n], "obs_mask": o["obs_mask"][:e],
                "prob": o["prob"][:e], "logodds": o["logodds"][:e]}
    return {"edge_offsets": dem.edge_offsets, "det_offsets": dem.det_offsets, "det_idx": dem.det_idx,
            "obs_mask": dem.obs_mask, "prob": dem.prob, "logodds": dem.logodds, "mech_class": dem.mech_class}


_ARRAYS = ("det_offsets", "det_idx", "obs_mask", "prob", "logodds")


def _run_serve(state):
    """Every patch is opened, submits `cycles` cycles (up to k of them between two steps), reads its requests'
    hyperedges and is closed."""
    srv, patches, level = state["srv"], state["patches"], state["level"]
    pids, ids = [], []
    for c, h, blocks, registered in patches:
        pid = srv.open_circuit_patch(c, h)
        pids.append(pid)
        ids.append([srv.register_cycle(pid, b) for b in blocks] if registered else None)
    got, owner = [[] for _ in patches], {}
    for t in range(state["cycles"]):
        for i, (c, h, blocks, registered) in enumerate(patches):
            if registered:
                rid = srv.submit_registered(pids[i], ids[i][min(t, 1)])
            else:
                rid = srv.submit(pids[i], blocks[t], final=False)
            owner[rid] = i
        if (t + 1) % state["k"] and t + 1 < state["cycles"]:
            continue
        while srv.step(level):
            pass
        for rid in srv.completed():
            got[owner[rid]].append(srv.result(rid))
            srv.release(rid)
    for pid in pids:
        srv.close_patch(pid)
    out = []
    for rs in got:
        rs.sort(key=lambda r: r["cycle"])
        d = {k: np.concatenate([r[k] for r in rs]) for k in _ARRAYS}
        d["obs_mask"] = d["obs_mask"].view(np.int64)
        d["det_offsets"] = d["det_offsets"].view(np.int32)
        d["det_idx"] = d["det_idx"].view(np.int32)
        out.append([d[k] for k in _ARRAYS])
    # one list per array keeps the number of outputs small
    return {k: np.concatenate([o[j] for o in out]) for j, k in enumerate(_ARRAYS)}


# -- work -----------------------------------------------------------------------------------------------------------

_NCOMP = {"L0": {32: 1, 33: 1, 34: 2, 35: 6}, "L1": {32: 1, 33: 1, 34: 3, 35: 10}, "L2": {32: 1, 33: 1, 34: 3, 35: 15}}
#: hyperedges per mechanism (about: counted on the listed circuits), and for the kinds that differ
_EDGES = {"L0": 0.17, "L1": 0.25, "L2": 0.26}
_EDGES_KIND = {"adaptive": 0.09, "repetition": 0.08, "z_only": 0.07}


def _mechanisms(ops, level):
    kinds = np.asarray(ops)[:, 0]
    return sum(n * int((kinds == k).sum()) for k, n in _NCOMP[level].items())


def work(case):
    level = case["level"]
    if case["kind"] == "serve":
        circs = []
        for c, h, blocks, registered in _serve_blocks(case, 0):
            circs += [blocks[min(t, 1)] if registered else blocks[t] for t in range(case["cycles"])]
        rows = [(b["ops"], b["recs"].size, b["n_locations"]) for b in circs]
    else:
        rows = [(c.ops, c.recs.size, c.n_locations) for c in _circuits(case)]
    total = 0.0
    for ops, n_recs, n_loc in rows:
        m = _mechanisms(ops, level)
        edges = m * _EDGES_KIND.get("z_only" if case.get("z_only") else case["kind"], _EDGES[level])
        # rows, record lookbacks and noise in; per hyperedge an offset, a mask, P, w and about three detectors out
        total += 16.0 * len(ops) + 4.0 * n_recs + 4.0 * n_loc + edges * (4 + 8 + 4 + 4 + 12)
        if case["kind"] == "bb_grad":
            total += 4.0 * n_loc + 8.0 * edges             # cotangents in, gradient out
        elif case.get("io") != "host" and case["kind"] != "serve":
            total += 4.0 * m                               # the class of every mechanism out
    return {"bytes": total, "flops": 0}


# -- exact values ---------------------------------------------------------------------------------------------------

# which planes a component XORs: bit 0 / 1 = an X / Z error on the first qubit, 2 / 3 on the second
_CODES = {32: [1], 33: [2], 34: [1, 2, 3], 35: [4, 8, 1, 5, 2, 10, 12, 9, 3, 6, 13, 7, 15, 11, 14]}
_CK = {32: (2.0, 1.0), 33: (2.0, 1.0), 34: (4.0 / 3.0, 2.0), 35: (16.0 / 15.0, 8.0)}


def _masks(ops, recs, n_qubits, level, keys, obs_keys):
    """(mask key of every mechanism, its location, its channel kind).  keys: one row per detector, obs_keys one per
    observable (uint64 pairs, or Python integers in one column)."""
    ops = np.asarray(ops, np.int64).reshape(-1, 4)
    recs = np.asarray(recs, np.int64)
    kinds = ops[:, 0]
    is_m = np.isin(kinds, (2, 3, 5, 6))
    n_before = np.cumsum(is_m) - is_m                    # measurements before each row
    zero = np.zeros_like(keys[:1]) if keys.dtype != object else np.array([[0]], object)
    mh = np.repeat(zero, int(is_m.sum()), axis=0)        # key each measurement record flips
    for rows, table in ((np.flatnonzero(kinds == 16), keys), (np.flatnonzero(kinds == 17), obs_keys)):
        n = ops[rows, 2]
        which = np.repeat(np.arange(rows.size), n)
        at = np.arange(n.sum()) - np.repeat(np.cumsum(n) - n, n) + np.repeat(ops[rows, 1], n)
        m = np.repeat(n_before[rows], n) - recs[at]
        val = table[which] if table is keys else table[ops[rows, 3][which]]
        np.bitwise_xor.at(mh, m, val)
    ncomp = np.zeros(len(ops), np.int64)
    for k, n in _NCOMP[level].items():
        ncomp[kinds == k] = n
    base = np.cumsum(ncomp) - ncomp
    out = np.repeat(zero, int(ncomp.sum()), axis=0)
    loc = np.repeat(ops[:, 3], ncomp)
    kind = np.repeat(kinds, ncomp)
    x = np.repeat(zero, n_qubits, axis=0)
    z = np.repeat(zero, n_qubits, axis=0)
    cut = np.flatnonzero(np.diff(kinds)) + 1             # runs of one row kind (gates of a run are disjoint)
    starts = np.concatenate([[0], cut])
    ends = np.concatenate([cut, [len(ops)]])
    for s, e in zip(starts[::-1], ends[::-1]):
        k = int(kinds[s])
        a, b = ops[s:e, 1], ops[s:e, 2]
        if k in (2, 3, 5, 6):
            w = mh[n_before[s:e]]
            if k == 2:
                x[a] ^= w
            elif k == 3:
                x[a], z[a] = w, zero
            elif k == 5:
                z[a] ^= w
            else:
                z[a], x[a] = w, zero
        elif k in (1, 4):
            x[a] = zero
            z[a] = zero
        elif k == 8:
            x[a], z[a] = z[a], x[a]
        elif k == 9:
            x[a] ^= z[a]
        elif k == 10:
            x[a] ^= x[b]
            z[b] ^= z[a]
        elif k == 11:
            x[a] ^= z[b]
            x[b] ^= z[a]
        elif k >= 32:
            two = k == 35
            p = [x[a], z[a]] + ([x[b], z[b]] if two else [])
            for c in range(_NCOMP[level][k]):
                code, w = _CODES[k][c], np.repeat(zero, e - s, axis=0)
                for j, plane in enumerate(p):
                    if code >> j & 1:
                        w = w ^ plane
                out[base[s:e] + c] = w
    return out, loc, kind


def _terms(kind, p):
    t, dt = np.zeros(p.size), np.zeros(p.size)
    for k, (c, n) in _CK.items():
        s = kind == k
        t[s] = -np.log1p(-c * p[s]) / n
        dt[s] = c / n / (1.0 - c * p[s])
    return t, dt


def _classes(circ, noise, level, seed=1):
    """64-bit P and w of one circuit's hyperedges in the order of their smallest mechanism, and per mechanism its
    hyperedge (-1: none), location and dt/dp."""
    r = np.random.default_rng(seed)
    keys = r.integers(1, 1 << 63, size=(max(circ.n_detectors, 1), 2), dtype=np.uint64)
    obs = r.integers(1, 1 << 63, size=(max(circ.n_observables, 1), 2), dtype=np.uint64)
    m, loc, kind = _masks(circ.ops, circ.recs, circ.n_qubits, level, keys, obs)
    live = np.flatnonzero((m != 0).any(axis=1) & (noise[loc] > 0))
    mm = np.ascontiguousarray(m[live])
    order = np.lexsort((mm[:, 1], mm[:, 0]))             # stable: equal masks stay in mechanism order
    s = mm[order]
    new = np.ones(order.size, bool)
    new[1:] = (s[1:] != s[:-1]).any(axis=1)
    group = np.cumsum(new) - 1
    first = order[new]
    rank = np.empty(first.size, np.int64)
    rank[np.argsort(first, kind="stable")] = np.arange(first.size)
    cls = np.full(loc.size, -1, np.int64)
    cls[live[order]] = rank[group]
    t, dt = _terms(kind, noise[loc])
    T = np.bincount(cls[live], weights=t[live], minlength=first.size)
    P = -np.expm1(-T) / 2
    return P, np.log1p(-P) - np.log(P), cls, loc, dt


def exact(case, seed):
    if case["kind"] == "serve":
        return _exact_serve(case, seed)
    circs = _circuits(case)
    noise = _noise(circs, seed).astype(np.float64)
    P, W, l0 = [], [], 0
    for c in circs:
        p, w, cls, loc, dt = _classes(c, noise[l0:l0 + c.n_locations], case["level"])
        P.append(p)
        W.append(w)
        l0 += c.n_locations
    P, W = np.concatenate(P), np.concatenate(W)
    if case["kind"] == "bb_grad":
        g = torch.Generator().manual_seed(int(seed))
        gp, gw = torch.randn(P.size, generator=g), 1e-3 * torch.randn(P.size, generator=g)
        gbar = gp.double().numpy() - gw.double().numpy() / (P * (1 - P))
        s = cls >= 0
        grad = np.bincount(loc[s], weights=(gbar * 0.5 * (1 - 2 * P))[cls[s]] * dt[s], minlength=noise.size)
        return {"prob": P, "logodds": W, "grad": grad}
    if case.get("io") == "host":
        return {"det_offsets": None, "det_idx": None, "obs_mask": None, "prob": P, "logodds": W}
    return {"edge_offsets": None, "det_offsets": None, "det_idx": None, "obs_mask": None, "prob": P, "logodds": W,
            "mech_class": None}


def _exact_serve(case, seed):
    """Request t of a patch delivers the hyperedges whose smallest detector lies in cycle t - H; over a stream they
    are those of the whole circuit.  Masks as Python integers (bit = detector), for their smallest detector."""
    P, W = [], []
    for c, h, blocks, registered in _serve_blocks(case, seed):
        allb = c.cycle_blocks()
        n_cycles = case["cycles"] + h + 1                # every mechanism of a delivered hyperedge lies in these
        noise = [blocks[min(t, len(blocks) - 1)]["noise"] if registered else
                 (blocks[t]["noise"] if t < len(blocks) else np.zeros(allb[t]["n_locations"])) for t in range(n_cycles)]
        noise += [np.zeros(b["n_locations"]) for b in allb[n_cycles:]]
        noise = np.concatenate([np.asarray(v, np.float64) for v in noise])
        D = c.n_detectors
        keys = np.array([[1 << j] for j in range(D)] or [[0]], object)
        obs = np.array([[1 << (D + j)] for j in range(max(c.n_observables, 1))], object)
        m, loc, kind = _masks(c.ops, c.recs, c.n_qubits, case["level"], keys, obs)
        t, _ = _terms(kind, noise[loc])
        sums, dets = {}, (1 << D) - 1
        for key, v in zip(m[:, 0], t):
            if key and v > 0:
                sums[key] = sums.get(key, 0.0) + v
        ends = np.cumsum([b["n_detectors"] for b in allb])
        at = [[] for _ in range(case["cycles"])]
        for key, v in sums.items():                      # in the order of the smallest mechanism
            low = key & dets
            if not low:
                continue
            cyc = int(np.searchsorted(ends, (low & -low).bit_length() - 1, side="right")) + h
            if cyc < case["cycles"]:
                at[cyc].append(v)
        T = np.array([v for part in at for v in part])
        p = -np.expm1(-T) / 2
        P.append(p)
        W.append(np.log1p(-p) - np.log(p))
    return {"det_offsets": None, "det_idx": None, "obs_mask": None, "prob": np.concatenate(P),
            "logodds": np.concatenate(W)}
