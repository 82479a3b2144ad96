"""Timing cases over the library's public entry points.

Each case is a dict of plain values; `prepare` makes what a program holds before
the call (gate lists, schedules, states on the GPU), `run` makes one pass, and
`exact` gives the same results in 64 bits from plain torch / numpy.  Kinds:

  circuit   |0...0> -> a supremacy circuit -> the state on the GPU
  cluster   a program's own clusters, one qs_apply_cluster call each
  diagonal  a CZ / T phase product and a table diagonal
  measure   statistics and sampled bitstrings of a state
  readout   probabilities, norm and single amplitudes of a state
  batch     many small circuits in one launch, statistics of each
  train     the cost model's network: epochs of full-batch training
"""
import math
import random

import numpy as np
import torch

from paper_1704_01127_gb300 import qs

# ---------------------------------------------------------------- the cases


def listed():
    return [
        # the smallest circuit in use, one op per gate (the plain form): latency and launches
        {"name": "plain_4x4_c128", "kind": "circuit", "rows": 4, "cols": 4, "cycles": 10, "dtype": "c128", "fuse": False,
         "remap": False},
        # a 20-qubit circuit fused into clusters: the state sits in L2, a few CTAs per sweep
        {"name": "circuit_4x5_c64", "kind": "circuit", "rows": 4, "cols": 5, "cycles": 25, "dtype": "c64", "fuse": True,
         "remap": False},
        # the headline workload: 30 qubits, 25 CZ cycles, complex128 (16 GiB)
        {"name": "circuit_5x6_c128", "kind": "circuit", "rows": 5, "cols": 6, "cycles": 25, "dtype": "c128", "fuse": True,
         "remap": False},
        # the bulk precision with qubits moved off the low index bits; reading the state moves them back
        {"name": "circuit_4x7_c64_remap", "kind": "circuit", "rows": 4, "cols": 7, "cycles": 25, "dtype": "c64",
         "fuse": True, "remap": True},
        # own clusters of every size on any qubits, both precisions, states well over L2
        {"name": "cluster_27_c128", "kind": "cluster", "n": 27, "dtype": "c128", "count": 5, "pick": 1},
        {"name": "cluster_28_c64", "kind": "cluster", "n": 28, "dtype": "c64", "count": 5, "pick": 2},
        # diagonal gates on their own (T and CZ layers, a 6-qubit table)
        {"name": "diagonal_27_c128", "kind": "diagonal", "n": 27, "dtype": "c128", "terms": 27, "k": 6, "pick": 3},
        # end of a run: output statistics and 2^20 bitstrings
        {"name": "measure_28_c128", "kind": "measure", "n": 28, "dtype": "c128", "draws": 1 << 20},
        # the same in complex64 with few bitstrings
        {"name": "measure_29_c64", "kind": "measure", "n": 29, "dtype": "c64", "draws": 4096},
        # reading results out: probabilities on the device, the norm, 2048 amplitudes to the host
        {"name": "readout_26_c64", "kind": "readout", "n": 26, "dtype": "c64", "count": 2048},
        # many small circuits (16-21 qubits) in one graph-replayed launch
        {"name": "batch_96_c64", "kind": "batch", "circuits": 96, "dtype": "c64", "k_max": 4, "pick": 4},
        # fitting the cost model: 20 epochs on 4096 timings
        {"name": "train_4096", "kind": "train", "rows": 4096, "epochs": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["circuit", "circuit", "circuit", "cluster", "cluster", "diagonal", "measure", "measure", "readout",
                       "batch", "train"])
    dtype = rng.choice(["c64", "c128"])
    big = 28 if dtype == "c64" else 27
    if kind == "circuit":
        while True:
            rows, cols = rng.randint(2, 5), rng.randint(3, 7)
            if 8 <= rows * cols <= 28:
                break
        fuse = rows * cols > 20 or rng.random() < 0.75   # the plain form is for small circuits
        return {"kind": kind, "rows": rows, "cols": cols, "cycles": rng.randint(8, 30), "dtype": dtype, "fuse": fuse,
                "remap": fuse and rows * cols >= 12 and rng.random() < 0.3}
    if kind == "cluster":
        return {"kind": kind, "n": rng.randint(10, big), "dtype": dtype, "count": rng.randint(1, 6),
                "pick": rng.randint(10, 10 ** 6)}
    if kind == "diagonal":
        n = rng.randint(10, big)
        return {"kind": kind, "n": n, "dtype": dtype, "terms": rng.randint(1, 2 * n), "k": rng.randint(1, 9),
                "pick": rng.randint(10, 10 ** 6)}
    if kind == "measure":
        return {"kind": kind, "n": rng.randint(8, big + 1), "dtype": dtype, "draws": _log(rng, 1, 1 << 20)}
    if kind == "readout":
        return {"kind": kind, "n": rng.randint(8, big), "dtype": dtype, "count": _log(rng, 1, 2048)}
    if kind == "batch":   # the batched workload is complex64
        return {"kind": kind, "circuits": _log(rng, 1, 96), "dtype": "c64", "k_max": rng.choice([3, 4, 5]),
                "pick": rng.randint(10, 10 ** 6)}
    return {"kind": kind, "rows": _log(rng, 64, 8192), "epochs": rng.randint(1, 20)}


# ------------------------------------------------------------------- inputs


def _gates(rows, cols, cycles, seed):
    """A supremacy circuit's gates, (cycle, name, qubits): H on every qubit, then CZ layers on a grid in eight
    staggered layouts; a qubit that had a CZ in the cycle before and has none now gets T the first time, later one
    of T, X^1/2, Y^1/2 other than its last."""
    rnd = random.Random(seed)
    layouts = [("h", 1, 0), ("v", 0, 0), ("h", 0, 0), ("v", 1, 0), ("v", 0, 1), ("h", 1, 1), ("v", 1, 1), ("h", 0, 1)]
    n = rows * cols
    out = [(0, "h", (q,)) for q in range(n)]
    busy, last = set(), {}
    for t in range(1, cycles + 1):
        way, a, b = layouts[(t - 1) % 8]
        pairs = []
        for r in range(rows):
            for c in range(cols):
                if way == "h" and c % 2 == a and r % 2 == b and c + 1 < cols:
                    pairs.append((r * cols + c, r * cols + c + 1))
                if way == "v" and r % 2 == a and c % 2 == b and r + 1 < rows:
                    pairs.append((r * cols + c, (r + 1) * cols + c))
        now = {q for p in pairs for q in p}
        for q in sorted(busy - now):
            last[q] = rnd.choice([g for g in ("t", "x_1_2", "y_1_2") if g != last[q]]) if q in last else "t"
            out.append((t, last[q], (q,)))
        out += [(t, "cz", p) for p in pairs]
        busy = now
    return n, out


def _batch_sizes(case):
    rnd = random.Random(case["pick"])
    return [rnd.choice([(4, 4), (4, 5), (3, 7)]) + (rnd.randint(8, 40),) for _ in range(case["circuits"])]


def _dtype(case):
    return (torch.complex64, qs.QS_C64) if case["dtype"] == "c64" else (torch.complex128, qs.QS_C128)


def _state(case, seed):
    """2^n complex Gaussian amplitudes of norm 1: what a deep random circuit leaves."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    psi = torch.empty(1 << case["n"], dtype=_dtype(case)[0], device="cuda")
    torch.view_as_real(psi).normal_(generator=g)
    return psi.mul_(1.0 / math.sqrt(2.0 * psi.numel()))


def _clusters(case, seed):
    """case["count"] clusters of 1..5 qubits: the qubits from the case, the unitaries from the seed."""
    rnd, g = random.Random(case["pick"]), np.random.Generator(np.random.PCG64(seed))
    out = []
    for i in range(case["count"]):
        k = (5, 3, 4, 1, 2, 5)[i % 6]
        z = g.standard_normal((1 << k, 1 << k)) + 1j * g.standard_normal((1 << k, 1 << k))
        q, r = np.linalg.qr(z)
        out.append((rnd.sample(range(case["n"]), k), q * (np.diag(r) / np.abs(np.diag(r)))))
    return out


def _diagonals(case, seed):
    """T-type coefficients and CZ pairs, and a table diagonal: the qubits from the case, the values from the seed."""
    rnd, g = random.Random(case["pick"]), np.random.Generator(np.random.PCG64(seed))
    n = case["n"]
    edges = [tuple(sorted(rnd.sample(range(n), 2))) for _ in range(case["terms"])]
    return g.integers(0, 8, n), edges, rnd.sample(range(n), case["k"]), np.exp(2j * np.pi * g.uniform(size=1 << case["k"]))


def _timings(case, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    X = g.standard_normal((case["rows"], qs.QS_NFEAT))
    Y = np.tanh(X @ g.standard_normal(qs.QS_NFEAT)) + 0.1 * g.standard_normal(case["rows"])
    W = 0.2 * g.standard_normal(12 * 64 + 64 + 64 * 64 + 64 + 64 + 1)
    return X, Y, W


class _Held:
    """Library handles that go with the Python object that holds them."""

    def __init__(self, **kw):
        self.frees = []
        self.__dict__.update(kw)

    def keep(self, handle, free):
        self.frees.append((free, handle))
        return handle

    def __del__(self):
        for free, handle in reversed(self.frees):
            free(handle)


class _Buffer:
    def __init__(self, owner, ptr, count, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (count,), "typestr": typestr, "data": (ptr, False), "version": 3}


def _seen(s, case):
    """The library's state as a tensor, in place."""
    n = qs.qs_num_qubits(s.h)
    typestr = "<c8" if case["dtype"] == "c64" else "<c16"
    return torch.as_tensor(_Buffer(s, qs.qs_device_ptr(s.h), 1 << n, typestr), device="cuda")


def prepare(case, seed):
    s = _Held(case=case)
    kind = case["kind"]
    if kind == "circuit":
        n, gates = _gates(case["rows"], case["cols"], case["cycles"], seed)
        dt = _dtype(case)[1]
        s.sched = s.keep(qs.qs_schedule_build(n, qs.gates_from_tuples(gates), fuse=case["fuse"], merge_phase=case["fuse"]),
                         qs.qs_schedule_free)
        if case["remap"]:
            qs.qs_schedule_remap(s.sched, qs.qs_schedule_choose_remap(s.sched, dt))
        qs.qs_schedule_upload(s.sched, dt)
        s.h = s.keep(qs.qs_alloc(n, dt), qs.qs_free)
    elif kind == "batch":
        scheds = []
        for i, (r, c, t) in enumerate(_batch_sizes(case)):
            n, gates = _gates(r, c, t, 1000 * seed + i)
            scheds.append(qs.qs_schedule_build(n, qs.gates_from_tuples(gates), k_max=case["k_max"], search_runs=1,
                                               search_first=1))
            if i == 0:
                s.n0 = n
        s.stream = torch.cuda.Stream()
        s.b = s.keep(qs.qs_batch_create(scheds, _dtype(case)[1], s.stream), qs.qs_batch_free)
        # what qs_batch_tune settles on for many circuits; a few are split over more threads each
        qs.qs_batch_set_config(s.b, *((4, 128) if case["circuits"] >= 32 else (8, 512)))
        for sc in scheds:
            qs.qs_schedule_free(sc)
    elif kind == "train":
        s.X, s.Y, s.W = _timings(case, seed)
        s.m = s.keep(qs.qs_mlp_create(0), qs.qs_mlp_free)
    else:
        s.psi = _state(case, seed)
        s.h = s.keep(qs.qs_wrap(s.psi, case["n"], _dtype(case)[1]), qs.qs_free)
        if kind == "cluster":
            s.clusters = _clusters(case, seed)
        elif kind == "diagonal":
            s.coeff, s.edges, s.qubits, s.table = _diagonals(case, seed)
        elif kind == "measure":
            s.seed = seed
        else:
            s.at = np.random.Generator(np.random.PCG64(seed)).integers(0, 1 << case["n"], case["count"]).astype(np.uint64)
            s.p = torch.empty(1 << case["n"], dtype=torch.float64, device="cuda")
    return s


# ----------------------------------------------------------------- one pass


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "circuit":
        qs.qs_init_basis(s.h, 0)
        qs.qs_run_circuit(s.h, s.sched)
        return _seen(s, case)
    if kind == "cluster":
        for qubits, U in s.clusters:
            qs.qs_apply_cluster(s.h, qubits, U)
        return s.psi
    if kind == "diagonal":
        qs.qs_apply_phase(s.h, s.coeff, s.edges)
        qs.qs_apply_diag(s.h, s.qubits, s.table)
        return s.psi
    if kind == "measure":
        bits, stats = qs.qs_sample_stats(s.h, s.seed, case["draws"])
        return {"bits": bits.view(np.int64), "stats": np.array(stats)}
    if kind == "readout":
        qs.qs_probabilities(s.h, s.p, out_on_device=True)
        return {"p": s.p, "norm": np.array(qs.qs_norm(s.h)), "at": qs.qs_get_amplitudes_at(s.h, s.at)}
    if kind == "batch":
        qs.qs_batch_run_graph(s.b)
        return {"stats": qs.qs_batch_stats(s.b, case["circuits"]), "first": qs.qs_batch_get_amplitudes(s.b, 0, s.n0)}
    qs.qs_mlp_set_params(s.m, s.W)
    loss = qs.qs_mlp_train(s.m, s.X, s.Y, case["epochs"])
    return {"loss": np.array(loss), "params": qs.qs_mlp_get_params(s.m)}


# ------------------------------------------------------- work and tolerance


def work(case):
    kind = case["kind"]
    amp = 8 if case.get("dtype") == "c64" else 16
    if kind == "circuit":
        # the state written once; 14 flops an amplitude for each dense one-qubit gate (about one per qubit every 6 cycles)
        n = case["rows"] * case["cols"]
        return {"bytes": amp << n, "flops": 14 * (n + n * case["cycles"] // 6) << n}
    if kind == "batch":
        n, flops = 0, 0
        for r, c, t in _batch_sizes(case):
            n += 1 << r * c
            flops += 14 * (r * c + r * c * t // 6) << r * c
        return {"bytes": amp * n, "flops": flops}
    if kind == "train":
        return {"bytes": 8 * case["rows"] * 13, "flops": 6 * case["epochs"] * case["rows"] * (12 * 64 + 64 * 64 + 64)}
    N = 1 << case["n"]
    if kind == "cluster":
        ks = [(5, 3, 4, 1, 2, 5)[i % 6] for i in range(case["count"])]
        return {"bytes": 2 * amp * N * len(ks), "flops": sum((8 << k) - 2 for k in ks) * N}
    if kind == "diagonal":
        return {"bytes": 4 * amp * N, "flops": 12 * N}
    if kind == "measure":
        return {"bytes": amp * N + 8 * case["draws"], "flops": 12 * N}
    return {"bytes": 2 * amp * N + 8 * N, "flops": 6 * N}


def tolerance(case):
    """About four times the error against `exact` that was measured over these ranges: complex64 circuits and clusters
    5e-7 (rounded FP32 sums), complex128 ones 1e-13 (47 bits of a group's largest amplitude per sweep); statistics
    5e-8 (complex64: each p rounded to 32 bits) and 1e-14; training 1e-15 after 20 epochs."""
    c64 = case.get("dtype") == "c64"
    kind = case["kind"]
    if kind == "train":
        return {"rel": 1e-11}
    if kind in ("measure", "readout"):   # bitstrings are whole numbers and do not differ
        return {"rel": 2e-7 if c64 else 1e-13}
    return {"rel": 2e-6 if c64 else 5e-13}


# ------------------------------------------------------------ 64-bit results

_H = math.sqrt(0.5)
_GATE = {"h": [[_H, _H], [_H, -_H]],
         "x_1_2": [[0.5 + 0.5j, 0.5 - 0.5j], [0.5 - 0.5j, 0.5 + 0.5j]],
         "y_1_2": [[0.5 + 0.5j, -0.5 - 0.5j], [0.5 + 0.5j, 0.5 + 0.5j]]}


def _simulate(n, gates):
    """The gates one by one on |0...0>, complex128."""
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1
    for _, name, qubits in gates:
        q = qubits[0]
        v = psi.view(-1, 2, 1 << q)
        if name == "t":
            v[:, 1] *= complex(_H, _H)
        elif name == "cz":
            a, b = sorted(qubits)
            psi.view(-1, 2, 1 << (b - a - 1), 2, 1 << a)[:, 1, :, 1].neg_()
        else:
            (a, b), (c, d) = _GATE[name]
            x, y = v[:, 0].clone(), v[:, 1].clone()
            v[:, 0] = a * x
            v[:, 0] += b * y
            v[:, 1] = c * x
            v[:, 1] += d * y
    return psi


def _stats(p):
    """sum p, -sum p ln p, mean of N p, mean of (N p)^2."""
    return torch.stack([p.sum(), -torch.special.xlogy(p, p).sum(), p.sum(), p.numel() * p.square().sum()])


def _exact_train(case, seed):
    X, Y, W = (torch.from_numpy(a).cuda() for a in _timings(case, seed))
    m, v = torch.zeros_like(W), torch.zeros_like(W)
    cuts = [12 * 64, 64, 64 * 64, 64, 64, 1]
    for t in range(1, case["epochs"] + 2):
        W1, b1, W2, b2, w3, b3 = torch.split(W, cuts)
        W1, W2 = W1.view(12, 64), W2.view(64, 64)
        a1 = torch.tanh(X @ W1 + b1)
        a2 = torch.tanh(a1 @ W2 + b2)
        e = a2 @ w3 + b3 - Y
        if t > case["epochs"]:
            return {"loss": e.square().mean(), "params": W}
        g = 2 * e / Y.numel()
        d2 = g[:, None] * w3 * (1 - a2 * a2)
        d1 = (d2 @ W2.T) * (1 - a1 * a1)
        G = torch.cat([(X.T @ d1).reshape(-1), d1.sum(0), (a1.T @ d2).reshape(-1), d2.sum(0), a2.T @ g, g.sum()[None]])
        m = 0.9 * m + 0.1 * G
        v = 0.999 * v + 0.001 * G * G
        W = W - 3e-3 * math.sqrt(1 - 0.999 ** t) / (1 - 0.9 ** t) * m / (torch.sqrt(v) + 1e-8)


def exact(case, seed):
    kind = case["kind"]
    if kind == "circuit":
        n, gates = _gates(case["rows"], case["cols"], case["cycles"], seed)
        return _simulate(n, gates)
    if kind == "batch":
        stats, first = [], None
        for i, (r, c, t) in enumerate(_batch_sizes(case)):
            psi = _simulate(*_gates(r, c, t, 1000 * seed + i))
            first = psi if first is None else first
            stats.append(_stats(torch.view_as_real(psi).square().sum(-1)))
        return {"stats": torch.stack(stats), "first": first}
    if kind == "train":
        return _exact_train(case, seed)
    psi = _state(case, seed).to(torch.complex128)
    if kind == "cluster":
        for qubits, U in _clusters(case, seed):
            axes = sorted(qubits, reverse=True)      # from the highest index bit down
            cuts = [case["n"]] + axes + [-1]
            dims = []
            for hi, lo in zip(cuts[:-2], cuts[1:-1]):
                dims += [1 << (hi - lo - 1), 2]
            dims.append(1 << axes[-1])
            at = [2 * axes.index(q) + 1 for q in reversed(qubits)]   # qubits[0] is the matrix index's lowest bit
            v = psi.view(dims).movedim(at, list(range(len(at))))
            w = torch.from_numpy(np.ascontiguousarray(U)).cuda() @ v.reshape(1 << len(at), -1)
            psi = w.view(v.shape).movedim(list(range(len(at))), at).reshape(-1)
        return psi
    if kind == "diagonal":
        coeff, edges, qubits, table = _diagonals(case, seed)
        w8 = [complex(1, 0), complex(_H, _H), 1j, complex(-_H, _H), -1, complex(-_H, -_H), -1j, complex(_H, -_H)]
        for q, c in enumerate(coeff):
            psi.view(-1, 2, 1 << q)[:, 1] *= w8[int(c) % 8]
        for a, b in edges:
            psi.view(-1, 2, 1 << (b - a - 1), 2, 1 << a)[:, 1, :, 1].neg_()
        x = torch.zeros(psi.numel(), dtype=torch.int64, device="cuda")
        i = torch.arange(psi.numel(), device="cuda")
        for j, q in enumerate(qubits):
            x |= ((i >> q) & 1) << j
        return psi * torch.from_numpy(table).cuda()[x]
    p = torch.view_as_real(psi).square().sum(-1)
    if kind == "measure":
        return {"bits": None, "stats": _stats(p)}
    at = np.random.Generator(np.random.PCG64(seed)).integers(0, 1 << case["n"], case["count"])
    return {"p": p, "norm": p.sum(), "at": psi[torch.from_numpy(at).cuda()]}
