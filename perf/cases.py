"""Performance cases of the reconstruction library: what a program that uses
it has it do, through the binding's public entry points.

A case is a dict of plain values.  ``kind`` names the entry point; a single
network is given by its cut edges ("up>down" subcircuit pairs) and the output
qubits of every subcircuit.  Tensors are pseudo-physical: every physical
variant of a subcircuit (3 measurement bases per upstream cut, 4 initial
states per downstream cut) is an exponential (Porter-Thomas-like)
distribution over its measured bits, put into the Pauli basis, so that the
reconstructed distribution sums to one as a real circuit's does."""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2502_03445_gb300 import tqc

# The 30-qubit grid shape of the benchmark: 4 subcircuits of width 10, 10 cuts.
GRID30_EDGES = "3>1 2>3 0>2 0>1 0>3 3>1 3>1 2>1 0>1 0>3"
GRID30_OUTS = "6,9,13,15,26|1,4,7,10,16,18,21,22,25,27|0,8,11,12,14,17,20,23|2,3,5,19,24,28,29"
# The cut 48-qubit QAOA circuit restricted to its bin of 2^24 states.
QAOA48_EDGES = ("0>2 0>2 0>2 4>0 0>1 1>3 0>3 3>2 3>4 1>2 4>3 0>1 1>4 0>4 1>3 2>4 4>1 3>2 0>3 4>2 4>3")
QAOA48_OUTS = "0,3,4,7,9|16,20|1,2,5,6,11,14|8,10,15,19,21,22|12,13,17,18,23"


def listed():
    scrambled = "0,1,2,4,5,7,8,9,12,13,15,17,19,20,23,27|3,6,10,11,14,16,18,21,22,24,25,26"
    return [
        # The smallest call: a 10-qubit line circuit cut once (two wire cuts),
        # its whole distribution; latency of one call.
        dict(name="line10", kind="contract", n=10, edges="0>1 1>0", outs="0,1,2,3,4|5,6,7,8,9", free=10, prec="auto",
             inp="f64", out="f32"),
        # A latency-critical loop that may not allocate: 15 qubits, 4
        # subcircuits, the caller's own device tensors.
        dict(name="noalloc15", kind="noalloc", n=15, edges="0>1 1>2 2>3 0>3 1>3",
             outs="0,4,9|1,5,7,13|2,6,10,14|3,8,11,12", free=15, prec="auto", inp="f64", out="f32"),
        # One bin of a streamed distribution: a mid-size network, 20 of 24
        # qubits free, other fixed bits than the plan's, FP64 results.
        dict(name="bin24_f64", kind="contract", n=24, edges="0>1 0>2 1>2 1>3 2>3 2>4 3>4 0>3 1>4",
             outs="3,8,12,19|0,6,14,20,22|1,5,10,16,23|2,7,11,17,21|4,9,13,15,18", free=20, prec="auto", inp="f64",
             out="f64"),
        # A mid-size full distribution with many subcircuits (many small
        # steps): 23 qubits, 6 subcircuits, FP32 tensors.
        dict(name="net23", kind="contract", n=23, edges="0>1 0>2 1>3 2>3 2>4 3>5 4>5 1>4 0>5 1>2",
             outs="2,9,15|0,7,12,20|1,5,11,18|3,8,13,21|4,10,16,19|6,14,17,22", free=23, prec="auto", inp="f32",
             out="f32"),
        # The headline: the 30-qubit grid shape, the full 2^30 distribution.
        dict(name="grid30", kind="contract", n=30, edges=GRID30_EDGES, outs=GRID30_OUTS, free=30, prec="auto",
             inp="f64", out="f32"),
        # The same network where only FP32 arithmetic will do, a quarter of it.
        dict(name="grid30_fp32", kind="contract", n=30, edges=GRID30_EDGES, outs=GRID30_OUTS, free=28, prec="fp32",
             inp="f64", out="f32"),
        # The largest: a bin of the 48-qubit QAOA network, tensor-bound,
        # sliced into a 32 GB budget.
        dict(name="qaoa48", kind="contract", n=24, edges=QAOA48_EDGES, outs=QAOA48_OUTS, free=24, prec="auto",
             inp="f64", out="f32", budget_gb=32),
        # Two subcircuits sharing two cuts, their qubits interleaved: the
        # Kronecker expansion dominates.
        dict(name="pair28", kind="contract", n=28, edges="0>1 0>1", outs=scrambled, free=28, prec="auto", inp="f64",
             out="f32"),
        # A list of one million arbitrary states of the 30-qubit network.
        dict(name="states1m", kind="states", n=30, edges=GRID30_EDGES, outs=GRID30_OUTS, count=1000000, inp="f64",
             out="f32"),
        # Many independent networks of uneven sizes in one call.
        dict(name="batch48", kind="batch", count=48, n_lo=16, n_hi=24, shapes=3000),
        # End to end from and to pinned host memory.
        dict(name="host26", kind="host", n=26, edges="0>1 0>2 1>2 1>3 2>3 0>3 0>1",
             outs="0,5,9,14,18,23|1,4,8,13,17,22,25|2,6,10,15,19,24|3,7,11,12,16,20,21", free=26, prec="auto",
             inp="f64", out="f32"),
        # Heavy state selection's first step: the norms of every output state.
        dict(name="norms30", kind="norms", n=30, edges=GRID30_EDGES, outs=GRID30_OUTS, inp="f64"),
    ]


# ------------------------------------------------------------------ drawing
def _edges(case):
    return [tuple(int(v) for v in e.split(">")) for e in case["edges"].split()]


def _outs(case):
    return [[int(q) for q in o.split(",")] if o else [] for o in case["outs"].split("|")]


def _sample(rng, n, m, cuts, width, node_bits, node_cuts=7):
    """(edges, outs) of a random connected acyclic cut network: subcircuit
    widths at most ``width``, node tensors of at most 2^node_bits entries; or
    None."""
    order = list(range(m))
    rng.shuffle(order)
    und = [(order[k], order[rng.randrange(k)]) for k in range(1, m)]
    while len(und) < cuts:
        und.append(tuple(rng.sample(range(m), 2)))
    rank = list(range(m))
    rng.shuffle(rank)
    edges = [(a, b) if rank[a] < rank[b] else (b, a) for a, b in und]
    up, down = [0] * m, [0] * m
    for a, b in edges:
        up[a] += 1
        down[b] += 1
    lo = [max(0, d - u) for u, d in zip(up, down)]
    hi = [min(width - u, node_bits - 2 * (u + d)) for u, d in zip(up, down)]
    if any(u + d > node_cuts or h < x for u, d, h, x in zip(up, down, hi, lo)) or not sum(lo) <= n <= sum(hi):
        return None
    o = list(lo)
    while sum(o) < n:
        j = rng.choice([j for j in range(m) if o[j] < hi[j]])
        o[j] += 1
    qs = list(range(n))
    rng.shuffle(qs)
    outs, at = [], 0
    for k in o:
        outs.append(sorted(qs[at:at + k]))
        at += k
    return edges, outs


def _order(edges, nfree, states=0):
    """The contraction order of fewest multiply-adds (dynamic programming over
    sets of subcircuits): ([(a, b)], multiply-adds, largest intermediate).
    ``states``: each step over at most that many distinct assignments of its
    output qubits."""
    m = len(nfree)
    cuts = [0] * (1 << m)
    q = [0] * (1 << m)
    for s in range(1, 1 << m):
        low = s & -s
        j = low.bit_length() - 1
        cuts[s] = cuts[s ^ low] ^ sum(1 << c for c, e in enumerate(edges) if j in e)
        q[s] = q[s ^ low] + nfree[j]
    best, split = [0] * (1 << m), [0] * (1 << m)
    for s in range(1, 1 << m):
        if s & (s - 1):
            low, t, got = s & -s, (s - 1) & s, []
            while t:
                if t & low:
                    c = 4 ** bin(cuts[t] | cuts[s ^ t]).count("1") * (min(2 ** q[s], states) if states else 2 ** q[s])
                    got.append((best[t] + best[s ^ t] + c, t))
                t = (t - 1) & s
            best[s], split[s] = min(got)
    steps, big = [], 0

    def tree(s):
        nonlocal big
        if not s & (s - 1):
            return s.bit_length() - 1
        if s != (1 << m) - 1:
            big = max(big, 2 ** (q[s] + 2 * bin(cuts[s]).count("1")))
        steps.append((tree(split[s]), tree(s ^ split[s])))
        return m + len(steps) - 1

    tree((1 << m) - 1)
    return steps, best[-1], big


def _text(edges, outs):
    return dict(edges=" ".join("%d>%d" % e for e in edges), outs="|".join(",".join(map(str, o)) for o in outs))


def _network(rng, n, ms, extra, width, node_bits, macs, big, node_cuts=7):
    """A random network of n qubits within the limits; or None."""
    for _ in range(300):
        m = rng.randint(*ms)
        got = _sample(rng, n, m, m - 1 + rng.randint(*extra), width, node_bits, node_cuts)
        if got is None:
            continue
        _, work, largest = _order(got[0], [len(o) for o in got[1]])
        if work <= macs and largest <= big:
            return got
    return None


def draw(rng):
    """One more case of the listed ones' ranges."""
    while True:
        kind = rng.choices(["contract", "pair", "states", "batch", "host", "noalloc", "norms"],
                           [45, 14, 12, 9, 8, 6, 6])[0]
        inp = rng.choice(["f64", "f64", "f32"])
        out = rng.choice(["f32", "f32", "f32", "f64"])
        if kind == "batch":
            lo = rng.randint(14, 20)
            return dict(kind="batch", count=round(2 ** rng.uniform(2, 5.9)), n_lo=lo, n_hi=lo + rng.randint(2, 5),
                        shapes=rng.randrange(1 << 20))
        if kind == "contract":
            n = rng.randint(10, 29)
            prec = rng.choices(["auto", "fp32", "bf16x3", "tf32"], [70, 14, 9, 7])[0]
            got = _network(rng, n, (2, 7), (0, 8), 14, 22, 2 ** (36 if prec == "fp32" else 39), 2 ** 30)
            if got is None:
                continue
            free = n if rng.random() < 0.6 else rng.randint(max(8, n - 10), n)
            return dict(kind="contract", n=n, **_text(*got), free=free, prec=prec, inp=inp, out=out)
        if kind == "pair":
            n = rng.randint(16, 28)
            got = _network(rng, n, (2, 2), (0, 1), 24, 27, 2 ** 36, 2 ** 30)
            if got is None:
                continue
            return dict(kind="contract", n=n, **_text(*got), free=n, prec="auto", inp=inp, out=out)
        if kind == "host":
            n = rng.randint(14, 26)
            got = _network(rng, n, (2, 5), (0, 4), 13, 22, 2 ** 36, 2 ** 29)
            if got is None:
                continue
            return dict(kind="host", n=n, **_text(*got), free=n, prec="auto", inp=inp, out="f32")
        if kind == "noalloc":
            n = rng.randint(8, 15)
            got = _network(rng, n, (2, 5), (0, 2), 9, 15, 2 ** 24, 2 ** 17)
            if got is None:
                continue
            return dict(kind="noalloc", n=n, **_text(*got), free=n, prec="auto", inp=inp, out=out)
        if kind == "states":
            n = rng.randint(16, 30)
            got = _network(rng, n, (3, 5), (1, 5), 11, 22, 2 ** 42, 2 ** 28, node_cuts=6)
            if got is None:
                continue
            count = round(10 ** rng.uniform(3, 6))
            per_state = _order(got[0], [0] * len(got[1]))
            if per_state[1] > 400000 or per_state[2] > 4 ** 6:
                continue
            return dict(kind="states", n=n, **_text(*got), count=count, inp=inp, out=out)
        n = rng.randint(12, 32)
        got = _network(rng, n, (2, 5), (0, 6), 14, 23, 2 ** 60, 2 ** 60)
        if got is None:
            continue
        return dict(kind="norms", n=n, **_text(*got), inp=inp)


def _batch_networks(case):
    rng, nets = random.Random(case["shapes"]), []
    while len(nets) < case["count"]:
        n = rng.randint(case["n_lo"], case["n_hi"])
        got = _network(rng, n, (2, 8), (0, 4), 12, 18, 2 ** 32, 2 ** 26)
        if got is not None:
            nets.append((n, *got))
    return nets


# ------------------------------------------------------------------ inputs
def _tensor(roles, n_out, gen):
    """One pseudo-physical node tensor, flat [c_0]..[c_k-1][x], FP64."""
    ups = [i for i, r in enumerate(roles) if r == 0]
    u, d = len(ups), len(roles) - len(ups)
    p = torch.empty((3 ** u * 4 ** d, 2 ** (u + n_out)), dtype=torch.float64, device="cuda")
    p.exponential_(generator=gen)
    p /= p.sum(1, keepdim=True)
    # [basis]*u [init]*d [y]*u [x] -> one Pauli axis per cut
    p = p.reshape((3,) * u + (4,) * d + (2,) * u + (2 ** n_out,))
    for t in range(u):  # measured bit: I = Z0 + Z1, X = X0 - X1, Y = Y0 - Y1, Z = Z0 - Z1 (bases Z, X, Y)
        b0, b1 = p.movedim((t, u + d + t), (0, 1)).unbind(1)
        z, x, y = range(3)
        e = torch.stack([b0[z] + b1[z], b0[x] - b1[x], b0[y] - b1[y], b0[z] - b1[z]])
        p = e.unsqueeze(1).movedim((0, 1), (t, u + d + t))  # the bit's axis keeps its place, now of length 1
    for t in range(d):  # initial states 0, 1, +, +i
        s0, s1, sp, si = p.unbind(u + t)
        p = torch.stack([s0 + s1, 2 * sp - s0 - s1, 2 * si - s0 - s1, s0 - s1], u + t)
    p = p.reshape((4,) * (u + d) + (2 ** n_out,))
    place, a, b = [], 0, u
    for r in roles:
        place.append(a if r == 0 else b)
        a, b = (a + 1, b) if r == 0 else (a, b + 1)
    return p.permute(place + [u + d]).reshape(-1)


def _nodes(n, edges, outs, seed, inp):
    """The network's nodes with their tensors on the GPU."""
    nodes = []
    for j, o in enumerate(outs):
        gen = torch.Generator(device="cuda").manual_seed(seed * 1009 + j)
        cuts = [(c, e.index(j)) for c, e in enumerate(edges) if j in e]
        data = _tensor([r for _, r in cuts], len(o), gen)
        nodes.append(SimpleNamespace(out_qubits=o, cut_ids=[c for c, _ in cuts], cut_role=[r for _, r in cuts],
                                     data=data.float() if inp == "f32" else data))
    return nodes


def _fixed(case, seed):
    """(free qubits, a bit for every qubit): the bin of a case."""
    free = list(range(case.get("free", case["n"])))
    bits = np.random.RandomState(seed % (1 << 31)).randint(0, 2, case["n"]).astype(np.uint8)
    return free, bits


def _states(case, seed):
    return np.random.RandomState(seed % (1 << 31)).randint(0, 1 << case["n"], case["count"]).astype(np.uint64)


def _handle(n, nodes, inp, shape_only=False):
    host = [SimpleNamespace(out_qubits=d.out_qubits, cut_ids=d.cut_ids, cut_role=d.cut_role,
                            data=None if shape_only else d.data.cpu().numpy()) for d in nodes]
    return tqc.Network(SimpleNamespace(n_qubits=n, nodes=host), dtype=tqc.F32 if inp == "f32" else tqc.F64,
                       shape_only=shape_only)


def _dtype(name):
    return torch.float64 if name == "f64" else torch.float32


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        handles, plans, outs = [], [], []
        for i, (n, edges, o) in enumerate(_batch_networks(case)):
            h = _handle(n, _nodes(n, edges, o, seed * 131 + i, "f64"), "f64")
            p = tqc.Plan(h)
            handles.append(h)
            plans.append(p)
            outs.append(torch.empty(p.out_elems, dtype=torch.float32, device="cuda"))
            p.contract(outs[-1])  # the batched call asks for one contract of each plan first
        return dict(kind=kind, nets=handles, plans=plans, outs=outs)
    nodes = _nodes(case["n"], _edges(case), _outs(case), seed, case["inp"])
    s = dict(kind=kind)
    s["net"] = net = _handle(case["n"], nodes, case["inp"], shape_only=kind == "noalloc")
    if kind == "norms":
        s["outs"] = [torch.empty(2 ** len(d.out_qubits), dtype=torch.float64, device="cuda") for d in nodes]
        return s
    if kind == "states":
        s["plan"] = tqc.Plan(net, free_qubits=[])
        s["states"] = _states(case, seed)
        s["out"] = torch.empty(case["count"], dtype=_dtype(case["out"]), device="cuda")
        return s
    free, bits = _fixed(case, seed)
    bin_ = {} if len(free) == case["n"] else {"free_qubits": free}
    s["plan"] = plan = tqc.Plan(net, precision=case["prec"], mem_budget=case.get("budget_gb", 0) << 30, **bin_)
    s["bits"] = bits if bin_ else None
    if kind == "host":
        s["tensors"] = [d.data.cpu().pin_memory() for d in nodes]
        s["inp"] = tqc.F32 if case["inp"] == "f32" else tqc.F64
        s["out"] = torch.empty(plan.out_elems, dtype=torch.float32, pin_memory=True)
        return s
    s["out"] = torch.empty(plan.out_elems, dtype=_dtype(case["out"]), device="cuda")
    if kind == "noalloc":
        s["tensors"] = [d.data for d in nodes]
        s["inp"] = tqc.F32 if case["inp"] == "f32" else tqc.F64
    return s


def run(state):
    kind = state["kind"]
    if kind == "contract":
        state["plan"].contract(state["out"], fixed_bits=state["bits"])
        return state["out"]
    if kind == "noalloc":
        state["plan"].contract_noalloc(state["tensors"], state["out"], in_dtype=state["inp"])
        return state["out"]
    if kind == "states":
        state["plan"].contract_states(state["states"], state["out"])
        return state["out"]
    if kind == "host":
        z = state["plan"].contract_host(state["tensors"], state["out"], in_dtype=state["inp"])
        return {"p": state["out"], "z": z}
    if kind == "norms":
        for j, o in enumerate(state["outs"]):
            state["net"].hss_norms(j, o)
        return state["outs"]
    tqc.contract_batch(state["plans"], state["outs"])
    return state["outs"]


# ------------------------------------------------------------------ what it takes
def work(case):
    if case["kind"] == "batch":
        total = [0, 0]
        for n, edges, outs in _batch_networks(case):
            w = work(dict(kind="contract", n=n, **_text(edges, outs), free=n, inp="f64", out="f32"))
            total = [total[0] + w["bytes"], total[1] + w["flops"]]
        return {"bytes": total[0], "flops": total[1]}
    edges, outs = _edges(case), _outs(case)
    isz, osz = (4 if case["inp"] == "f32" else 8), (8 if case.get("out") == "f64" else 4)
    deg = [sum(j in e for e in edges) for j in range(len(outs))]
    full = [4 ** c * 2 ** len(o) for c, o in zip(deg, outs)]
    if case["kind"] == "norms":
        return {"bytes": isz * sum(full) + 8 * sum(2 ** len(o) for o in outs), "flops": 2 * sum(full)}
    if case["kind"] == "states":
        macs = _order(edges, [len(o) for o in outs], case["count"])[1]
        return {"bytes": isz * sum(full) + (8 + osz) * case["count"], "flops": 2 * macs}
    nfree = [sum(q < case["free"] for q in o) for o in outs]
    elems = sum(4 ** c * 2 ** f for c, f in zip(deg, nfree))
    return {"bytes": isz * elems + osz * 2 ** case["free"], "flops": 2 * _order(edges, nfree)[1]}


# ------------------------------------------------------------------ exact values
def _digits(places, bits):
    """Offsets of every value of a string of fields (lowest first), each of
    ``bits`` bits placed at a multiple of ``places[i]``."""
    off = torch.zeros(1, dtype=torch.int64, device="cuda")
    for p in places:
        d = torch.arange(1 << bits, dtype=torch.int64, device="cuda") * p
        off = (d[:, None] + off[None, :]).reshape(-1)
    return off


def _matrix(f, rows, cols):
    """Factor (qubits, cuts, flat [x][cuts]) as [x, open cuts] x [shared cuts]."""
    qs, cs, v = f
    x = torch.arange(1 << len(qs), dtype=torch.int64, device="cuda") << (2 * len(cs))
    r = (x[:, None] + _digits([4 ** cs.index(c) for c in rows], 2)[None, :]).reshape(-1)
    return v[r[:, None] + _digits([4 ** cs.index(c) for c in cols], 2)[None, :]]


def _pair(f, g):
    shared = [c for c in f[1] if c in g[1]]
    fo, go = [c for c in f[1] if c not in shared], [c for c in g[1] if c not in shared]
    v = _matrix(f, fo, shared) @ _matrix(g, go, shared).T
    v = v.reshape(1 << len(f[0]), 4 ** len(fo), 1 << len(g[0]), 4 ** len(go)).permute(2, 0, 3, 1)
    return f[0] + g[0], fo + go, v.reshape(-1)


def _factor(d, n_fixed=(), bits=None):
    """A node as a factor [x over its free outputs][cuts], 64 bits."""
    k, qs = len(d.cut_ids), d.out_qubits
    free = [q for q in qs if q not in n_fixed]
    base = sum(int(bits[q]) << qs.index(q) for q in qs if q in n_fixed)
    x = _digits([1 << qs.index(q) for q in free], 1) + base
    e = _digits([4 ** (k - 1 - i) << len(qs) for i in range(k)], 2)
    return free, list(d.cut_ids), d.data.double()[(x[:, None] + e[None, :]).reshape(-1)]


def _reduce(edges, fs, keep=1):
    steps = _order(edges, [len(f[0]) for f in fs])[0]
    for a, b in steps[:len(fs) - keep]:
        fs.append(_pair(fs[a], fs[b]))
        fs[a] = fs[b] = None
    return [f for f in fs if f is not None]


def _mass(edges, nodes):
    fs = []
    for d in nodes:
        q, c, v = _factor(d)
        fs.append(([], c, v.reshape(1 << len(q), -1).sum(0)))
    return _reduce(edges, fs)[0][2][0]


def _exact_bin(n, edges, nodes, free, bits):
    (qs, _, v), = _reduce(edges, [_factor(d, set(range(n)) - set(free), bits) for d in nodes])
    v = v / _mass(edges, nodes)
    place = [1 << free.index(q) for q in qs]
    low = min(len(qs), 15)
    lo, hi = _digits(place[:low], 1), _digits(place[low:], 1)
    out = torch.empty_like(v)
    for i in range(0, len(hi), 1024):
        out[(hi[i:i + 1024, None] + lo[None, :]).reshape(-1)] = v[i << low:(i + len(hi[i:i + 1024])) << low]
    return out


def exact(case, seed):
    if case["kind"] == "batch":
        return [_exact_bin(n, e, _nodes(n, e, o, seed * 131 + i, "f64"), list(range(n)), None)
                for i, (n, e, o) in enumerate(_batch_networks(case))]
    edges, outs = _edges(case), _outs(case)
    if case["kind"] in ("contract", "host", "noalloc"):
        if _order(edges, [sum(q < case["free"] for q in o) for o in outs])[1] > 2 ** 41:
            return None  # minutes of 64-bit arithmetic
    nodes = _nodes(case["n"], edges, outs, seed, case["inp"])
    if case["kind"] == "norms":
        return [d.data.double().reshape(-1, 2 ** len(d.out_qubits)).square().sum(0).sqrt() for d in nodes]
    if case["kind"] == "states":
        f, g = _reduce(edges, [_factor(d) for d in nodes], keep=2)
        a, b = _matrix(f, [], f[1]), _matrix(g, [], f[1])
        st = torch.from_numpy(_states(case, seed).astype(np.int64)).cuda()
        xa, xb = (sum(((st >> q) & 1) << i for i, q in enumerate(h[0])) for h in (f, g))
        p = torch.cat([(a[xa[i:i + 65536]] * b[xb[i:i + 65536]]).sum(1) for i in range(0, len(st), 65536)])
        return p / _mass(edges, nodes)
    free, bits = _fixed(case, seed)
    p = _exact_bin(case["n"], edges, nodes, free, bits)
    if case["kind"] != "host":
        return p
    return {"p": p, "z": float(_mass(edges, nodes)) * 0.5 ** len(edges)}
