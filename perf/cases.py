"""Performance cases: what users of this framework have it do, through its public entry points.

A pass advances a network by a number of 50-us time steps (or trains the rate-function
surrogate, or computes one step's gap currents); every state is a network of its own, so
passes on one state continue the same simulation, as a program's step loop does.

`work` counts one time step as the unit that cannot be saved: a step reads the 15 words of
a cell that the update needs and writes the 18 it produces, reads each stored connection
(2 bytes of column, 4 more where it has a weight of its own; 4 bytes per matrix entry) and
evaluates each pair.  Initial states, graphs and weights are seeded; `exact` is the same
computation in 64 bits, in plain torch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1612_01501_gb300 import ion

DT = 0.05
PAIR_FLOPS = 7      # the junction term without its exponential, summed up
CELL_FLOPS = 380    # one cell's update
_stream = None


def listed():
    return [
        # the closed loop of the paper's real-time mode: every step takes the evoked input from
        # the host and gives the axon voltages back; the smallest calls, latency counts
        {"name": "loop_1003", "kind": "loop", "n": 1003, "steps": 20},
        # the 64-cell all-to-all network, in one persistent launch: step latency
        {"name": "dense_64", "kind": "dense", "n": 64, "steps": 1000, "persistent": True},
        # a mid-size all-to-all network with an odd size and a step count that is no multiple
        # of the captured graph's
        {"name": "dense_2999", "kind": "dense", "n": 2999, "steps": 120},
        # the 8192-cell all-to-all network of the benchmark
        {"name": "dense_8192", "kind": "dense", "n": 8192, "steps": 100},
        # 65 536 cells, random symmetric connectivity, short rows and rows of about 100
        {"name": "csr_65536_k10", "kind": "csr", "n": 65536, "k": 10, "steps": 100},
        {"name": "csr_65536_k100", "kind": "csr", "n": 65536, "k": 100, "steps": 100},
        # user-programmed connectivity: long rows, every connection with a weight of its own
        {"name": "csr_9001_k1000_weighted", "kind": "csr", "n": 9001, "k": 1000, "steps": 50, "weighted": True},
        # the whole connectivity matrix stored
        {"name": "matrix_8192", "kind": "matrix", "n": 8192, "steps": 25},
        # uncoupled cells: the update alone, larger than the caches
        {"name": "cells_2097401", "kind": "cells", "n": 2097401, "steps": 50},
        # a parameter sweep: many small networks of uneven sizes and kinds, the states read back
        {"name": "batch_96", "kind": "batch", "nets": 96, "sweep": 1000, "steps": 200},
        # the learned rate functions in the cell update, on the k = 100 network's size
        {"name": "surrogate_65536_k100", "kind": "surrogate", "n": 65536, "k": 100, "steps": 50},
        # fitting the rate functions: forward, backward and optimiser, the default batch
        {"name": "train_65536", "kind": "train", "samples": 65536, "epochs": 2, "batch": 1024},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    kind = rng.choice(["loop", "dense", "dense", "dense", "csr", "csr", "csr", "cells", "matrix", "batch",
                       "surrogate", "train"])
    if kind == "loop":
        return {"kind": kind, "n": _log_int(rng, 64, 10000), "steps": rng.randint(10, 20)}
    if kind == "dense":
        n = _log_int(rng, 48, 18688)
        c = {"kind": kind, "n": n, "steps": rng.randint(20, 120)}
        if n <= 144:
            c.update(persistent=True, steps=rng.randint(200, 1000))
        elif rng.random() < 0.2:   # linear junctions: the sum is O(n)
            c.update(linear=True, n=_log_int(rng, 145, 1_211_904))
        return c
    if kind == "csr":
        k = _log_int(rng, 4, 1000)
        c = {"kind": kind, "n": _log_int(rng, max(200, 2 * k), min(65536, 9_000_000 // k)), "k": k, "steps": rng.randint(20, 100)}
        if rng.random() < 0.3:
            c["weighted"] = True
        if rng.random() < 0.25:
            c["linear"] = True
        return c
    if kind == "cells":
        return {"kind": kind, "n": _log_int(rng, 1 << 14, 1 << 21), "steps": rng.randint(20, 50)}
    if kind == "matrix":
        return {"kind": kind, "n": _log_int(rng, 512, 8192), "steps": rng.randint(10, 25)}
    if kind == "batch":
        return {"kind": kind, "nets": rng.randint(12, 96), "sweep": rng.randint(1001, 9999), "steps": rng.randint(50, 200)}
    if kind == "surrogate":
        return {"kind": kind, "n": _log_int(rng, 2000, 65536), "k": _log_int(rng, 10, 100), "steps": rng.randint(20, 50)}
    batch = rng.choice([256, 512, 1024, 2048])
    return {"kind": "train", "samples": batch * rng.randint(16, 64) + rng.randint(0, 127), "epochs": 1, "batch": batch}


# ---- inputs --------------------------------------------------------------------------

def _gen(seed, what):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + what)


def _rand(seed, what, *shape, dtype=torch.float64):
    return torch.rand(*shape, generator=_gen(seed, what), device="cuda", dtype=dtype)


def _weight(g_ref, neighbours):
    """Per-junction weight at the same total coupling as 64 partners of weight g_ref."""
    return float(np.float32(g_ref * 64.0 / neighbours))


def _graph(n, k, seed, what=1):
    """Random symmetric graph, mean degree about k: sorted rows, no self loops (row_ptr, row, col on the GPU)."""
    half = max(1, k // 2)
    src = torch.arange(n, device="cuda").repeat_interleave(half)
    dst = torch.clamp((_rand(seed, what, n * half) * (n - 1)).long(), max=n - 2)
    dst = dst + (dst >= src)
    key = torch.unique(torch.cat([src * n + dst, dst * n + src]))
    row, col = key // n, key % n
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return row_ptr, row, col


def _edge_weights(g, n, row, col, seed):
    """One weight per junction (the same in both directions), g times a value in [0.5, 1.5)."""
    h = (torch.minimum(row, col) * n + torch.maximum(row, col) + 7919 * (int(seed) % 100_000)) * 2654435761
    u = ((h >> 13) & 0xFFFFFF).double() / float(1 << 24)
    return (g * (0.5 + u)).float()


def _csr(case, seed):
    n, k = case["n"], case["k"]
    row_ptr, row, col = _graph(n, k, seed)
    g = _weight(0.04, k)
    w = _edge_weights(g, n, row, col, seed) if case.get("weighted") else torch.full((len(col),), g, device="cuda")
    return row_ptr, row, col, w


def _initial(n, seed):
    """Rest state with the dendrites spread over +-5 mV (19 x n, FP32)."""
    S = torch.zeros(19, n, dtype=torch.float64, device="cuda")
    S[0:3] = -60.0
    S[3] = 3.715
    S[16] = 0.68
    r = _rates(S)
    for f, gate in ((4, "r"), (5, "s"), (6, "q"), (7, "k"), (8, "l"), (9, "ms"), (10, "hs"), (11, "ns"), (12, "xs"),
                    (13, "ma"), (14, "ha"), (15, "xa")):
        S[f] = r[gate][0]
    S[17] = 4.5 * S[4] ** 2 * (S[0] - 120.0)
    S[0] += 10.0 * _rand(seed, 2, n) - 5.0
    return S.float()


def _pulses(n, seed):
    """6 uA/cm^2 to about a fifth of the cells, steps 10 to 210."""
    cells = torch.nonzero(_rand(seed, 3, n) < 0.2).flatten().cpu().numpy().astype(np.int32)
    m = len(cells)
    return cells, np.full(m, 10, np.int64), np.full(m, 210, np.int64), np.full(m, 6.0, np.float32)


def _sweep(case):
    """Sizes, kinds, degrees and couplings of a sweep's networks."""
    rng = random.Random(case["sweep"])
    out = []
    for b in range(case["nets"]):
        n, g = _log_int(rng, 32, 4096), rng.uniform(0.01, 0.08)
        out.append((n, None, g) if b % 2 == 0 else (n, min(rng.randint(8, 256), n - 1), g))
    return out


def _surrogate(seed):
    """Weights of a rate-function MLP: seeded hidden layers, the output layer fitted by least squares."""
    rng = np.random.default_rng(int(seed) + 17)
    w1, b1 = rng.normal(0, 1.5, (64, 2)), rng.normal(0, 1.0, 64)
    w2, b2 = rng.normal(0, 0.18, (64, 64)), rng.normal(0, 0.1, 64)
    lo, hi = math.log(1.0), math.log(20.0)
    V = rng.uniform(-100, 50, 4096)
    lc = rng.uniform(lo, hi, 4096)
    x = np.stack([(V + 25.0) / 75.0, (lc - 0.5 * (lo + hi)) / (0.5 * (hi - lo))], 1)
    t = _targets(torch.from_numpy(V), torch.from_numpy(np.exp(lc))).numpy()
    shift, scale = t.mean(0), np.maximum(t.std(0), 1e-3)
    H = np.concatenate([np.tanh(np.tanh(x @ w1.T + b1) @ w2.T + b2), np.ones((4096, 1))], 1)
    sol = np.linalg.solve(H.T @ H + 0.1 * np.eye(65), H.T @ ((t - shift) / scale))
    p = {"w1": w1, "b1": b1, "w2": w2, "b2": b2, "w3": sol[:64].T, "b3": sol[64]}
    p = {k: np.asarray(v, np.float32) for k, v in p.items()}
    norm = {"in_shift": np.float32([-25.0, 0.5 * (lo + hi)]), "in_scale": np.float32([1 / 75.0, 2 / (hi - lo)]),
            "out_shift": shift.astype(np.float32), "out_scale": scale.astype(np.float32)}
    return p, norm


def _shared_stream():
    """One stream for every network of the process: their work runs in order."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream.cuda_stream


def prepare(case, seed):
    kind, s = case["kind"], {"case": case}
    stream = _shared_stream()
    if kind == "train":
        s["seed"] = int(seed)
        return s
    if kind == "batch":
        nets, states, pulses, off = [], [], [], 0
        for b, (n, k, g_ref) in enumerate(_sweep(case)):
            if k is None:
                nets.append(dict(n=n, kind=ion.DENSE_UNIFORM, g=_weight(g_ref, n)))
            else:
                row_ptr, _, col = _graph(n, k, seed, 100 + b)
                nets.append(dict(n=n, kind=ion.CSR, row_ptr=row_ptr.int().cpu().numpy(), col=col.int().cpu().numpy(),
                                 w=np.full(len(col), _weight(g_ref, k), np.float32)))
            off += n
        state = _initial(off, seed).cpu().numpy()
        s["h"] = _Handle(ion.ion_create_batch(nets, init_state=state, stream=stream))
        s["n"] = off
        ion.ion_set_input(s["h"].h, _pulses(off, seed))
        return s
    n = case["n"]
    kw = dict(init_state=_initial(n, seed).cpu().numpy(), stream=stream)
    flags = ion.FLAG_KAHAN | (ion.FLAG_SGJ if case.get("linear") else 0)
    if kind in ("dense", "loop"):
        if case.get("persistent"):
            flags |= ion.FLAG_PERSISTENT
        sim = ion.Simulation(n, ion.DENSE_UNIFORM, g=_weight(0.04, n), flags=flags, **kw)
    elif kind in ("csr", "surrogate"):
        row_ptr, _, col, w = _csr(case, seed)
        if kind == "surrogate":
            p, norm = _surrogate(seed)
            kw.update(surrogate=ion.weights_from_dict(p, **norm))
            flags |= ion.FLAG_SURROGATE
        sim = ion.Simulation(n, ion.CSR, row_ptr=row_ptr.int().cpu().numpy(), col=col.int().cpu().numpy(),
                             w=w.cpu().numpy(), flags=flags, **kw)
    elif kind == "matrix":
        W = _matrix(n, seed)
        torch.cuda.synchronize()   # the handle copies the matrix on its own stream
        sim = ion.Simulation(n, ion.DENSE_MATRIX, w=W, flags=flags, **kw)
    else:
        sim = ion.Simulation(n, ion.NO_GJ, flags=flags, **kw)
    s["sim"] = sim
    if kind == "loop":
        s["v"] = kw["init_state"][2].copy()
    else:
        sim.set_input(_pulses(n, seed))
    return s


def _matrix(n, seed):
    return (_weight(0.04, n) * 2.0 * _rand(seed, 5, n, n, dtype=torch.float32)).contiguous()


class _Handle:
    """A batch's handle, destroyed with the state."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        ion.ion_destroy(self.h)


class _Rows:
    """Rows of the device state as an array; keeps the network alive."""

    def __init__(self, sim, ptr, shape, row_bytes):
        self.sim = sim
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f4", "data": (ptr, False), "version": 3,
                                         "strides": (row_bytes, 4)}


def _device_state(sim):
    """The state's own buffers: V_dend (its current slot) and the 18 other fields."""
    v = ion.ion_state_device_ptr(sim.h, 0)
    a, b = ion.ion_state_device_ptr(sim.h, 1), ion.ion_state_device_ptr(sim.h, 2)
    return {"V_dend": torch.as_tensor(_Rows(sim, v, (1, sim.n), b - a), device="cuda"),
            "other": torch.as_tensor(_Rows(sim, a, (18, sim.n), b - a), device="cuda")}


def run(state):
    case = state["case"]
    kind, steps = case["kind"], case.get("steps")
    if kind == "train":
        w, loss = ion.ion_surrogate_train(n_samples=case["samples"], epochs=case["epochs"], batch=case["batch"],
                                          seed=state["seed"], stream=_shared_stream())
        out = {f: np.frombuffer(getattr(w, f), np.float32) for f in
               ("w1", "b1", "w2", "b2", "w3", "b3", "out_shift", "out_scale")}
        out["loss"] = loss
        return out
    if kind == "batch":
        ion.ion_step(state["h"].h, steps)
        return ion.ion_read_state(state["h"].h, state["n"])
    sim = state["sim"]
    if kind == "loop":   # an evoked input from the axons' last voltages, every step
        trace = np.empty((steps, sim.n), np.float32)
        v = state["v"]
        for t in range(steps):
            sim.step(1, dense=((np.float32(-55.0) - v) * np.float32(0.1))[None])
            v = sim.state(ion.FIELD["V_axon"])
            trace[t] = v
        state["v"] = v
        return {"V_axon": trace, "state": sim.state()}
    sim.step(steps)
    return _device_state(sim)


def work(case):
    kind, steps = case["kind"], case.get("steps", 1)
    cell_bytes = 4 * (15 + 18)
    if kind == "train":
        batches = case["samples"] // case["batch"] * case["epochs"]
        macs = 2 * 64 + 64 * 64 + 64 * 24
        return {"bytes": batches * case["batch"] * 26 * 4, "flops": batches * case["batch"] * macs * 2 * 3}
    if kind == "batch":
        cells = sum(n for n, _, _ in _sweep(case))
        pairs = sum(n * n if k is None else n * k for n, k, _ in _sweep(case))
        edges = sum(n * k for n, k, _ in _sweep(case) if k is not None)
        return {"bytes": steps * (cells * cell_bytes + 2 * edges) + 76 * cells,
                "flops": steps * (pairs * PAIR_FLOPS + cells * CELL_FLOPS)}
    n = case["n"]
    pairs, conn = 0, 0
    if kind in ("dense", "loop"):
        pairs = n if case.get("linear") else n * n
    elif kind == "matrix":
        pairs, conn = n * n, 4 * n * n
    elif kind in ("csr", "surrogate"):
        pairs = n * max(2, case["k"] // 2 * 2)
        conn = pairs * (6 if case.get("weighted") else 2)
    flops = pairs * PAIR_FLOPS + n * CELL_FLOPS
    if kind == "surrogate":
        flops += n * 3 * 2 * (2 * 64 + 64 * 64 + 64 * 24)
    if kind == "loop":
        cell_bytes += 8   # the evoked input in, the axon voltage out
    return {"bytes": steps * (n * cell_bytes + conn), "flops": steps * flops}


# ---- the same in 64 bits --------------------------------------------------------------

def _rise(V, vh, k):
    return torch.sigmoid((V - vh) / k)


def _fall(V, vh, k):
    return torch.sigmoid((vh - V) / k)


def _z_over_expm1(z):
    return torch.where(z == 0, torch.ones_like(z), z / torch.expm1(z))


def _rates_dend(V, ca):
    a = 1.7 * _rise(V, 5.0, 13.9)
    b = 0.1 * _z_over_expm1((V + 8.5) / 5.0)
    s = torch.clamp(2.0e-5 * ca, max=0.01)
    return {"r": (a / (a + b), (a + b) / 5.0), "s": (s / (s + 0.015), s + 0.015),
            "q": (_fall(V, -80.0, 4.0), torch.exp(-0.086 * V - 14.6) + torch.exp(0.070 * V - 1.87))}


def _rate_x(V):
    a = 1.3 * _z_over_expm1(-(V + 25.0) / 10.0)
    b = 1.69 * torch.exp(-0.0125 * (V + 35.0))
    return a / (a + b), a + b


def _rates_soma(V):
    one = torch.ones_like(V)
    return {"k": (_rise(V, -61.0, 4.2), one),
            "l": (_fall(V, -85.5, 8.5),
                  1.0 / (20.0 * torch.exp((V + 160.0) / 30.0) / (1.0 + torch.exp((V + 84.0) / 7.3)) + 35.0)),
            "ms": (_rise(V, -30.0, 5.5), 0 * one),
            "hs": (_fall(V, -70.0, 5.8), torch.exp((V + 40.0) / 33.0) / 3.0),
            "ns": (_rise(V, -3.0, 10.0), 1.0 / (5.0 + 47.0 * torch.exp((V + 50.0) / 900.0))),
            "xs": _rate_x(V)}


def _rates_axon(V):
    return {"ma": (_rise(V, -30.0, 5.5), torch.zeros_like(V)),
            "ha": (_fall(V, -60.0, 5.8), torch.exp((V + 40.0) / 33.0) / 1.5), "xa": _rate_x(V)}


def _rates(S):
    return {**_rates_dend(S[0], S[3]), **_rates_soma(S[1]), **_rates_axon(S[2])}


GATES = ("r", "s", "q", "k", "l", "ms", "hs", "ns", "xs", "ma", "ha", "xa")


def _targets(V, ca):
    """logit(x_inf) (at most 15 in size) and ln(tau) of every gate, interleaved."""
    r = {**_rates_dend(V, ca), **_rates_soma(V), **_rates_axon(V)}
    out = []
    for g in GATES:
        x = torch.clamp(r[g][0], min=1e-30, max=1.0)
        top = 1.0 - 2.0 ** -23   # 1 - 1e-7 in FP32
        out.append(torch.clamp(torch.log(x) - torch.log1p(-torch.clamp(x, max=top)), -15.0, 15.0))
        out.append(torch.zeros_like(V) if g in ("ms", "ma") else -torch.log(r[g][1]))
    return torch.stack(out, 1)


def _learned(S, p, norm):
    """All gates' rates from the MLP, one evaluation per compartment."""
    t = {k: torch.from_numpy(v).to("cuda", torch.float64) for k, v in {**p, **norm}.items()}
    out = {}
    for V, gates in ((S[0], ("r", "s", "q")), (S[1], ("k", "l", "ms", "hs", "ns", "xs")), (S[2], ("ma", "ha", "xa"))):
        x = (torch.stack([V, torch.log(S[3])], 1) - t["in_shift"]) * t["in_scale"]
        h = torch.tanh(torch.tanh(x @ t["w1"].T + t["b1"]) @ t["w2"].T + t["b2"])
        y = (h @ t["w3"].T + t["b3"]) * t["out_scale"] + t["out_shift"]
        for g in gates:
            i = GATES.index(g)
            out[g] = (torch.sigmoid(y[:, 2 * i]), torch.exp(-y[:, 2 * i + 1]))
    return out


def _euler(S, ic, iapp, rates):
    """One explicit-Euler step of every cell (19 x n, 64 bits)."""
    vd, vs, va, ca = S[0], S[1], S[2], S[3]
    r, s, q, k, l, hs, ns, xs, ha, xa, gcal = (S[f] for f in (4, 5, 6, 7, 8, 10, 11, 12, 14, 15, 16))
    ms, ma = rates["ms"][0], rates["ma"][0]
    icah = 4.5 * r * r * (vd - 120.0)
    N = torch.empty_like(S)
    N[0] = vd + DT * (iapp - icah - 35.0 * s * (vd + 75.0) - 0.125 * q * (vd + 43.0) - 0.016 * (vd - 10.0)
                      - 0.13 / 0.75 * (vd - vs) - ic)
    N[1] = vs - DT * (gcal * k ** 3 * l * (vs - 120.0) + 150.0 * ms ** 3 * hs * (vs - 55.0) + 9.0 * ns ** 4 * (vs + 75.0)
                      + 5.0 * xs ** 4 * (vs + 75.0) + 0.016 * (vs - 10.0) + 0.13 / 0.25 * (vs - vd)
                      + 0.13 / 0.85 * (vs - va))
    N[2] = va - DT * (240.0 * ma ** 3 * ha * (va - 55.0) + 20.0 * xa ** 4 * (va + 75.0) + 0.016 * (va - 10.0)
                      + 0.13 / 0.15 * (va - vs))
    N[3] = ca + DT * (-3.0 * icah - 0.075 * ca)
    for f, g in ((4, "r"), (5, "s"), (6, "q"), (7, "k"), (8, "l"), (10, "hs"), (11, "ns"), (12, "xs"), (14, "ha"),
                 (15, "xa")):
        N[f] = S[f] + DT * rates[g][1] * (rates[g][0] - S[f])
    N[9], N[13], N[16], N[17], N[18] = ms, ma, gcal, icah, ic
    return N


def _junction(d, linear):
    return d if linear else (0.8 * torch.exp(d * d * -0.01) + 0.2) * d


def _dense_current(V, g, linear=False):
    if linear:
        return g * (len(V) * V - V.sum())
    return torch.cat([(g * _junction(v[:, None] - V[None], False)).sum(1) for v in V.split(max(1, (1 << 27) // len(V)))])


def _csr_current(V, row_ptr, row, col, w, linear=False):
    return torch.zeros_like(V).index_add_(0, row, w * _junction(V[row] - V[col], linear))


def _exact_train(case, seed):
    n, B = case["samples"], case["batch"]
    M = (1 << 64) - 1

    def mix(z):
        z = z.astype(np.uint64)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))

    def uniform(base, m):
        k = np.arange(1, m + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        return (mix(k + np.uint64(base & M)) >> np.uint64(11)).astype(np.float64) / 9007199254740992.0

    def mix1(z):
        return int(mix(np.array([z & M], np.uint64))[0])

    def dev(a):
        return torch.from_numpy(np.asarray(a, np.float64)).cuda()

    lo, hi = float(np.log(np.float32(1.0))), float(np.log(np.float32(20.0)))
    V = dev((-100.0 + 150.0 * uniform(mix1(seed + 0x9E3779B97F4A7C15), n)).astype(np.float32))
    ca = dev(np.exp(lo + (hi - lo) * uniform(mix1(seed + 2 * 0x9E3779B97F4A7C15), n)).astype(np.float32))
    T = _targets(V, ca)
    mask = torch.ones(24, dtype=torch.float64, device="cuda")
    mask[[11, 19]] = 0.0   # the instantaneous gates have no time constant
    shift = T.mean(0) * mask
    scale = torch.where(mask > 0, torch.clamp(T.std(0, unbiased=False), min=1e-3), torch.ones_like(mask))
    T = (T - shift) / scale
    X = torch.stack([(V + 25.0) / 75.0, (torch.log(ca) - 0.5 * (lo + hi)) / (0.5 * (hi - lo))], 1)
    u = 2.0 * uniform(mix1(seed + 3), 5912) - 1.0
    shapes = {"w1": (64, 2), "b1": (64,), "w2": (64, 64), "b2": (64,), "w3": (24, 64), "b3": (24,)}
    fan, P, at = {"w1": 66, "w2": 128, "w3": 88}, {}, 0
    for f, sh in shapes.items():
        size = int(np.prod(sh))
        a = math.sqrt(6.0 / fan[f]) if f in fan else 0.0
        P[f] = dev((u[at:at + size] * a).reshape(sh).astype(np.float32))
        at += size
    m = {f: torch.zeros_like(p) for f, p in P.items()}
    v = {f: torch.zeros_like(p) for f, p in P.items()}
    per, step, loss = n // B, 0, 0.0
    total = per * case["epochs"]
    for ep in range(case["epochs"]):
        mul = int(0.6180339887498949 * n) + 2 * ((seed + ep) % 97) + 1
        while math.gcd(mul, n) != 1:
            mul += 1
        for b in range(per):
            i = torch.from_numpy((mul * np.arange(b * B, (b + 1) * B, dtype=np.int64) + (ep * 7919) % n) % n).cuda()
            x = X[i]
            h1 = torch.tanh(x @ P["w1"].T + P["b1"])
            h2 = torch.tanh(h1 @ P["w2"].T + P["b2"])
            e = (h2 @ P["w3"].T + P["b3"] - T[i]) * mask
            if ep == case["epochs"] - 1:
                loss += float((e * e).sum()) / (B * 22.0)
            d3 = 2.0 * e / (B * 22.0)
            d2 = (d3 @ P["w3"]) * (1.0 - h2 * h2)
            d1 = (d2 @ P["w2"]) * (1.0 - h1 * h1)
            g = {"w1": d1.T @ x, "b1": d1.sum(0), "w2": d2.T @ h1, "b2": d2.sum(0), "w3": d3.T @ h2, "b3": d3.sum(0)}
            lr = 1e-3 * (0.01 + 0.99 * 0.5 * (1.0 + math.cos(math.pi * (step / (total - 1) if total > 1 else 1.0))))
            step += 1
            for f in P:
                m[f] = 0.9 * m[f] + 0.1 * g[f]
                v[f] = 0.999 * v[f] + 0.001 * g[f] * g[f]
                P[f] = P[f] - lr * (m[f] / (1 - 0.9 ** step)) / (torch.sqrt(v[f] / (1 - 0.999 ** step)) + 1e-8)
    out = {f: p.flatten() for f, p in P.items()}
    out.update(out_shift=shift, out_scale=scale, loss=loss / per)
    return out


def exact(case, seed):
    kind, steps = case["kind"], case.get("steps")
    seed = int(seed)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "batch":
        parts, off = [], 0
        for b, (n, k, g_ref) in enumerate(_sweep(case)):
            parts.append((off, n, _weight(g_ref, n), None) if k is None
                         else (off, n, _weight(g_ref, k), _graph(n, k, seed, 100 + b)))
            off += n
        n = off

        def current(V):
            return torch.cat([_dense_current(V[o:o + c], g) if net is None else
                              _csr_current(V[o:o + c], *net, g) for o, c, g, net in parts])
    else:
        n = case["n"]
        linear = bool(case.get("linear"))
        if kind in ("dense", "loop"):
            def current(V):
                return _dense_current(V, _weight(0.04, n), linear)
        elif kind in ("csr", "surrogate"):
            row_ptr, row, col, w = _csr(case, seed)
            w = w.double()

            def current(V):
                return _csr_current(V, row_ptr, row, col, w, linear)
        elif kind == "matrix":
            W = _matrix(n, seed).double()

            def current(V):
                return (W * _junction(V[:, None] - V[None], False)).sum(1)
        else:
            def current(V):
                return torch.zeros_like(V)
    S = _initial(n, seed).double()
    pulsed = torch.zeros(n, dtype=torch.float64, device="cuda")
    if kind != "loop":
        pulsed[torch.from_numpy(_pulses(n, seed)[0]).long().cuda()] = 6.0
    net = _surrogate(seed) if kind == "surrogate" else None
    trace = []
    for t in range(steps):
        iapp = 0.1 * (-55.0 - S[2]) if kind == "loop" else (pulsed if 10 <= t < 210 else 0.0 * pulsed)
        S = _euler(S, current(S[0]), iapp, _learned(S, *net) if net else _rates(S))
        if kind == "loop":
            trace.append(S[2])
    if kind == "batch":
        return S
    if kind == "loop":
        return {"V_axon": torch.stack(trace), "state": S}
    return {"V_dend": S[0:1], "other": S[1:]}
