"""The engine's workloads as measurable cases: inputs, one pass, the work it cannot do without, and its
value in 64 bits.

Families (each a user's program around the public entry points):
  circuit    amplitudes of a random circuit on a grid (closed, with open qubits, sliced): tn_plan + tn_contract_slices
  dynamics   <Z> of a kicked-Ising evolution on a square, honeycomb or triangular lattice: tn_contract, or its graph form
  spinglass  ln Z of a +-J Ising model on a square lattice, real forms with exponent scaling
  mis        maximum weight of an independent set of a King's subgraph (max-plus semiring)
  ensemble   many small networks in one launch (tn_batch_*): Ising disorder ensembles, independent sets
  state      two-qubit gates on a state vector kept in a shuffled qubit order (one large leaf, open output)
  pair       one dense pairwise contraction of any extents, in every arithmetic form
  serve      a burst of small requests queued together on a server (host inputs, host results)
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2606_01852_gb300 as tn
from tn_inputs import circuits, greedy, ising_pf, kicked_ising, kings, workloads
from tn_inputs.network import Network, Path

COMPLEX = ("fp32", "tf32", "3xtf32", "bf16x3", "bf16x3m")
REAL = ("r32_fp32", "r32_tf32", "r32_3xtf32")
# the 13-cycle circuit's eight sliced labels (what the greedy slicer picks on its path) as text
SLICED_13 = "209,319,374,343,240,311,328,42"
SLICED_14 = ",".join(str(x) for x in workloads.RC40C14_SLICED)


def listed():
    return [
        # one amplitude of a 12-qubit circuit: the smallest call, nothing but latency
        dict(name="amplitude_12q", family="circuit", rows=3, cols=4, cycles=8, open=0, prec="fp32", seed=0, alpha=1.0,
             temperature=0.0, sliced="", count=1),
        # 16 correlated amplitudes of a 20-qubit circuit: small steps and a few tensor-core ones
        dict(name="amplitudes_20q_open", family="circuit", rows=4, cols=5, cycles=12, open=4, prec="3xtf32", seed=0,
             alpha=0.5, temperature=0.0, sliced="", count=1),
        # eight slices of the 13-cycle 40-qubit amplitude as one device pass: mid-size steps, large outputs
        dict(name="slices_40q_13", family="circuit", rows=5, cols=8, cycles=13, open=0, prec="bf16x3", seed=0, alpha=1.0,
             temperature=0.05, sliced=SLICED_13, count=8),
        # two slices of the 14-cycle 40-qubit amplitude: the largest dense steps
        dict(name="slices_40q_14", family="circuit", rows=5, cols=8, cycles=14, open=0, prec="bf16x3",
             seed=workloads.RC40C14_PATH["seed"], alpha=workloads.RC40C14_PATH["alpha"],
             temperature=workloads.RC40C14_PATH["temperature"], sliced=SLICED_14, count=2),
        # a long path of mostly tiny steps, replayed from a CUDA graph
        dict(name="dynamics_4x4", family="dynamics", rows=4, cols=4, steps=10, lattice="square", prec="3xtf32", seed=1,
             alpha=1.0, temperature=0.05, graph=True),
        # the plain FP32 form on the CUDA cores (the form others are checked against)
        dict(name="dynamics_5x5_fp32", family="dynamics", rows=5, cols=5, steps=2, lattice="square", prec="fp32", seed=1,
             alpha=0.0, temperature=0.05, graph=False),
        # a partition function far beyond FP32's range, real tensor-core form with exponent scaling
        dict(name="spinglass_20x20", family="spinglass", rows=20, cols=20, prec="r32_3xtf32", seed=1, alpha=0.0),
        # combinatorial optimisation: the max-plus semiring, exact integers
        dict(name="mis_16x16", family="mis", side=16, graph_seed=1, seed=3, alpha=0.0, temperature=0.05),
        # a disorder ensemble: thousands of small uneven networks in one launch
        dict(name="ensemble_ising_4096", family="ensemble", kind="ising", count=4096, pool=64, low=20, high=60),
        # a gate layer on a 26-qubit state: permutation, streaming steps, a large open output
        dict(name="state_26q", family="state", qubits=26, gates=4, layout_seed=26, prec="fp32"),
        # one dense contraction with ragged extents
        dict(name="pair_ragged_tf32", family="pair", m=3001, n=1999, k=1500, prec="tf32"),
        # queued small requests, packed by the server
        dict(name="serve_burst_128", family="serve", amplitudes=96, partitions=32, pool=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        case = _draw_one(rng)
        if case["family"] not in ("circuit", "dynamics", "spinglass", "mis"):
            return case
        # a path cheaper than the largest listed case, and intermediates a plan can hold several of
        net, path, sliced = _network(_key(case))
        flops = greedy.path_log2_flops(net, path, sliced) + math.log2(case.get("count", 1))
        if flops <= 36.0 and greedy.path_peak(net, path, sliced) <= 27:
            return case


def _draw_one(rng):
    family = rng.choice(("circuit",) * 3 + ("dynamics",) * 2 + ("pair",) * 2 +
                        ("spinglass", "mis", "ensemble", "state", "serve"))
    if family == "circuit":
        n_sliced = rng.choice((0, 0, 1, 2, 3, 4))
        return dict(family=family, rows=rng.randint(3, 5), cols=rng.randint(4, 6), cycles=rng.randint(6, 14),
                    open=rng.randint(0, 5), prec=rng.choice(COMPLEX), seed=rng.randint(0, 99),
                    alpha=rng.choice((0.5, 1.0)), temperature=0.0, sliced="greedy:%d" % n_sliced, count=2 ** n_sliced)
    if family == "dynamics":
        return dict(family=family, rows=rng.randint(3, 5), cols=rng.randint(3, 5), steps=rng.randint(2, 12),
                    lattice=rng.choice(kicked_ising.LATTICES), prec=rng.choice(COMPLEX), seed=rng.randint(0, 99),
                    alpha=rng.choice((0.5, 1.0)), temperature=0.0, graph=rng.random() < 0.5)
    if family == "spinglass":
        return dict(family=family, rows=rng.randint(8, 19), cols=rng.randint(8, 19), prec=rng.choice(REAL),
                    seed=rng.randint(0, 99), alpha=rng.choice((0.0, 1.0)))
    if family == "mis":
        return dict(family=family, side=rng.randint(8, 16), graph_seed=rng.randint(0, 99), seed=rng.randint(0, 99),
                    alpha=0.0, temperature=0.0)
    if family == "ensemble":
        kind = rng.choice(("ising", "ising", "mis"))
        low, high = rng.choice(((20, 40), (20, 60))) if kind == "ising" else rng.choice(((4, 5), (4, 7)))
        return dict(family=family, kind=kind, count=_log_int(rng, 64, 4096 if kind == "ising" else 1024),
                    pool=rng.randint(8, 48), low=low, high=high)
    if family == "state":
        return dict(family=family, qubits=rng.randint(12, 26), gates=rng.randint(1, 8), layout_seed=rng.randint(0, 999),
                    prec="fp32")
    if family == "serve":
        return dict(family=family, amplitudes=_log_int(rng, 8, 160), partitions=_log_int(rng, 4, 64),
                    pool=rng.randint(4, 16))
    return dict(family=family, m=_log_int(rng, 1, 6000), n=_log_int(rng, 1, 6000), k=_log_int(rng, 8, 6000),
                prec=rng.choice(COMPLEX + REAL))


# ---- networks ------------------------------------------------------------------------------------

def _key(case):
    return tuple(sorted((k, v) for k, v in case.items() if k != "name"))


def _couplings(case, seed):
    """The dynamics' (J, h), around the values the dynamics family is quoted on."""
    rng = np.random.Generator(np.random.PCG64(seed))
    return float(rng.uniform(0.8, 1.2)), float(rng.uniform(0.7, 1.1))


def _open_qubits(case):
    n = case["rows"] * case["cols"]
    return tuple(range(n - case["open"], n))


def _structure(case, seed):
    """The network of `seed` (labels and shapes do not depend on the seed)."""
    f = case["family"]
    if f == "circuit":
        return circuits.amplitude_network(case["rows"], case["cols"], case["cycles"], seed,
                                          open_qubits=_open_qubits(case))
    if f == "dynamics":
        J, h = _couplings(case, seed)
        return kicked_ising.expectation_network(case["rows"], case["steps"], J, h, 0.25, cols=case["cols"],
                                                lattice=case["lattice"])
    if f == "spinglass":
        return ising_pf.lattice_network(case["rows"], case["cols"], 0.44, seed=seed)
    if f == "mis":
        net = kings.kings_network(case["side"], 0.8, case["graph_seed"], "tropical")
        weights = np.random.Generator(np.random.PCG64(seed)).integers(1, 10, size=net.n_tensors)
        net.tensors = [np.where(t == 1.0, float(w), t) for t, w in zip(net.tensors, weights)]
        return net
    if f == "state":
        n = case["qubits"]
        rng = np.random.Generator(np.random.PCG64(case["layout_seed"]))
        wire = list(range(n))
        modes = [tuple(int(q) for q in rng.permutation(n))]
        label = n
        tensors = [None]
        gates = np.random.Generator(np.random.PCG64(seed))
        for _ in range(case["gates"]):
            a, b = (int(q) for q in rng.choice(n, size=2, replace=False))
            modes.append((label, label + 1, wire[a], wire[b]))
            wire[a], wire[b] = label, label + 1
            label += 2
            tensors.append(circuits.haar_unitary(gates).reshape(2, 2, 2, 2))
        return Network(tensors, modes, {x: 2 for x in range(label)}, tuple(wire))
    return Network([None, None], [(0, 2), (1, 2)], {0: case["m"], 1: case["n"], 2: case["k"]}, (0, 1))  # pair


@functools.lru_cache(maxsize=None)
def _network(key):
    """(network of seed 0, path, sliced labels) of a case."""
    case = dict(key)
    net = _structure(case, 0)
    if case["family"] == "state":
        return net, circuits.state_path(net), ()
    if case["family"] == "pair":
        return net, Path([(0, 1)]), ()
    path = greedy.greedy_path(net, case["seed"], case["alpha"], case.get("temperature", 0.0))
    text = case.get("sliced", "")
    if text.startswith("greedy:"):
        sliced = tuple(greedy.greedy_slicer(net, path, -1.0, max_slices=int(text[7:])))
    else:
        sliced = tuple(int(x) for x in text.split(",") if x)
    return net, path, sliced


def _real(case):
    return case["family"] in ("spinglass", "mis") or case.get("prec", "").startswith("r32")


def _inputs(case, seed):
    """The leaves of `seed` as the device tensors a program holds (complex64 or float32)."""
    net = _structure(case, seed)
    dtype = torch.float32 if _real(case) else torch.complex64
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    out = []
    for t, modes in zip(net.tensors, net.modes):
        if t is None:  # a large Gaussian tensor, unit variance per element
            shape = tuple(net.extent[x] for x in modes)
            out.append(torch.randn(int(np.prod(shape)), dtype=dtype, device="cuda", generator=gen).reshape(shape))
        else:
            out.append(torch.tensor(np.asarray(t), dtype=dtype, device="cuda"))
    return out


# ---- ensembles -----------------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _pool(kind, pool, low, high):
    """`pool` graphs as (network, path, incident edges, edges)."""
    out = []
    for g in range(pool):
        rng = np.random.Generator(np.random.PCG64(7 * g + 3))
        if kind == "ising":
            net = ising_pf.random_3regular_network(2 * int(rng.integers(low // 2, high // 2 + 1)), 100 + g)
        else:
            net = kings.kings_network(int(rng.integers(low, high + 1)), 0.8, 100 + g, "tropical")
        out.append((net, greedy.greedy_path(net, 0, 0.0)))
    return out


def _ensemble_leaves(kind, net, seed, rows):
    """Leaf tensors (rows, ...) of `rows` instances on one graph: couplings J = +-1 at beta = 0.5 (as the package's
    Ising networks fold them into the vertices), or vertex weights 1-9."""
    rng = np.random.Generator(np.random.PCG64(seed))
    if kind == "mis":
        w = rng.integers(1, 10, size=(rows, net.n_tensors)).astype(np.float64)
        return [np.where(t[None] == 1.0, w[:, u].reshape((rows,) + (1,) * t.ndim), t[None])
                for u, t in enumerate(net.tensors)]
    edges = net.meta["edges"]
    J = rng.choice(np.array([-1.0, 1.0]), size=(rows, len(edges)))
    out = []
    for u, es in enumerate(net.modes):
        t = 0.0
        for s in (0, 1):
            w = np.ones((rows,) + (2,) * len(es))
            for ax, e in enumerate(es):
                if edges[e][0] == u:
                    f = np.exp(0.5 * J[:, e, None] * (1 - 2 * s) * np.array([1.0, -1.0]))
                else:
                    f = np.broadcast_to(np.array([1.0, 0.0]) if s == 0 else np.array([0.0, 1.0]), (rows, 2))
                w = w * f.reshape((rows,) + (1,) * ax + (2,) + (1,) * (len(es) - 1 - ax))
            t = t + w
        out.append(t)
    return out


def _ensemble_members(case):
    """Graph of every network, and for each graph the networks on it."""
    of = np.arange(case["count"]) % case["pool"]
    return of, [np.nonzero(of == g)[0] for g in range(case["pool"])]


# ---- the serving burst ---------------------------------------------------------------------------

class _Serving:
    """A server with its plans, closed when the program drops it."""

    def __init__(self, plans):
        self.plans = plans
        self.server = tn.Server(max_inflight=8, n_streams=4, hbm_budget_bytes=8 << 30, pack_max=256)

    def __del__(self):
        self.server.destroy()
        for p in self.plans:
            p.destroy()


@functools.lru_cache(maxsize=None)
def _serve_nets(pool):
    net = circuits.amplitude_network(3, 4, 8, 12)
    return (net, greedy.greedy_path(net, 0, 1.0)), _pool("ising", pool, 20, 60)


def _serve_requests(case, seed):
    """[(plan index, leaves)]: amplitudes of one circuit with a bitstring each, then partition functions."""
    (net, _), pool = _serve_nets(case["pool"])
    rng = np.random.Generator(np.random.PCG64(seed))
    gates = [np.asarray(t, dtype=np.complex64) for t in circuits.amplitude_network(3, 4, 8, seed % 1000).tensors]
    out = []
    for _ in range(case["amplitudes"]):
        leaves = list(gates)
        for q in range(12):
            e = np.zeros(2, dtype=np.complex64)
            e[rng.integers(0, 2)] = 1.0
            leaves[len(leaves) - 12 + q] = e
        out.append((0, leaves))
    for j in range(case["partitions"]):
        g = j % case["pool"]
        leaves = _ensemble_leaves("ising", pool[g][0], seed * 1000 + j, 1)
        out.append((1 + g, [np.ascontiguousarray(t[0], dtype=np.float32) for t in leaves]))
    return out


# ---- prepare / run -------------------------------------------------------------------------------

def prepare(case, seed):
    f = case["family"]
    if f == "ensemble":
        pool = _pool(case["kind"], case["pool"], case["low"], case["high"])
        of, members = _ensemble_members(case)
        batch = tn.Batch([pool[g][0] for g in of], [pool[g][1] for g in of], complex_=False,
                         exp_scaling=case["kind"] == "ising",
                         semiring="standard" if case["kind"] == "ising" else "maxplus")
        first = np.concatenate([[0], np.cumsum([pool[g][0].n_tensors for g in of])])
        offsets = np.asarray(batch.leaf_offsets)
        packed = np.empty(batch.leaf_offsets[-1], dtype=np.float32)
        for g, rows in enumerate(members):
            if len(rows) == 0:
                continue
            for u, t in enumerate(_ensemble_leaves(case["kind"], pool[g][0], seed * 64 + g, len(rows))):
                t = t.reshape(len(rows), -1)
                packed[offsets[first[rows] + u][:, None] + np.arange(t.shape[1])] = t
        packed = torch.tensor(packed, device="cuda")
        values = torch.zeros((case["count"], 2), dtype=torch.float64, device="cuda")
        logs = torch.zeros(case["count"], dtype=torch.float64, device="cuda")
        batch.autotune(packed, values, logs)
        return dict(family=f, kind=case["kind"], batch=batch, packed=packed, values=values, logs=logs)
    if f == "serve":
        (net, path), pool = _serve_nets(case["pool"])
        plans = [tn.Plan(net, path, prec="3xtf32")]
        plans += [tn.Plan(n, p, prec="r32_3xtf32", exp_scaling=True) for n, p in pool]
        requests = _serve_requests(case, seed)
        return dict(family=f, serving=_Serving(plans), requests=[(plans[i], leaves) for i, leaves in requests],
                    amplitudes=np.zeros(case["amplitudes"], dtype=np.complex128),
                    partitions=np.zeros((case["partitions"], 2), dtype=np.float64))
    net, path, sliced = _network(_key(case))
    plan = tn.Plan(net, path, sliced, prec="r32_fp32" if f == "mis" else case["prec"], exp_scaling=f == "spinglass",
                   semiring="maxplus" if f == "mis" else "standard", max_slice_batch=case.get("count", 0))
    dtype = torch.float64 if _real(case) else torch.complex128
    out = torch.zeros(tuple(net.extent[x] for x in net.open_modes), dtype=dtype, device="cuda")
    log_scale = torch.zeros(1, dtype=torch.float64, device="cuda")
    return dict(family=f, plan=plan, inputs=_inputs(case, seed), out=out, log_scale=log_scale,
                graph=case.get("graph", False), count=case.get("count", 0))


def run(state):
    f = state["family"]
    if f == "ensemble":
        state["batch"].contract(state["packed"], state["values"], state["logs"], graph=True)
        if state["kind"] == "mis":
            return state["values"]
        return torch.log(state["values"][:, 0]) + state["logs"]  # ln Z
    if f == "serve":
        server, n = state["serving"].server, len(state["amplitudes"])
        tickets = server.submit_batch(state["requests"])
        for j, t in enumerate(tickets):
            if j < n:
                tn.check(server.poll(t, state["amplitudes"][j:j + 1]))
            else:
                row = state["partitions"][j - n]
                tn.check(server.poll(t, row[0:1], row[1:2]))
        z = state["partitions"]
        return {"amplitudes": state["amplitudes"].copy(), "ln_z": np.log(z[:, 0]) + z[:, 1]}
    if f == "circuit":
        state["plan"].contract_slices(state["inputs"], 0, state["count"], state["out"])
    elif state["graph"]:
        state["plan"].contract_graph(state["inputs"], state["out"])
    else:
        state["plan"].contract(state["inputs"], state["out"], state["log_scale"])
    if f == "spinglass":
        return torch.log(state["out"]) + state["log_scale"]  # ln Z
    return state["out"]


# ---- the work of a pass --------------------------------------------------------------------------

def _path_products(net, path, sliced):
    """(products of the steps every slice shares, products of one slice's own steps), one per term of a step."""
    ext, cut, keep = net.extent, set(sliced), set(net.open_modes)
    sets = [(frozenset(x for x in m if x not in cut), bool(cut & set(m))) for m in net.modes]
    shared = own = 0.0
    for i, j in path.pairs:
        (a, da), (b, db) = sets[i], sets[j]
        terms = float(np.prod([float(ext[x]) for x in a | b])) if a | b else 1.0
        if da or db:
            own += terms
        else:
            shared += terms
        sets.append((frozenset((a ^ b) | (a & b & keep)), da or db))
    return shared, own


def _net_work(net, path, sliced, count, real):
    shared, own = _path_products(net, path, sliced)
    elems = sum(float(np.prod([float(net.extent[x]) for x in m])) for m in net.modes)
    out = float(np.prod([float(net.extent[x]) for x in net.open_modes])) if net.open_modes else 1.0
    return ((4.0 if real else 8.0) * elems + (8.0 if real else 16.0) * out,
            (2.0 if real else 8.0) * (shared + own * count))


def work(case):
    f = case["family"]
    if f == "ensemble":
        of, members = _ensemble_members(case)
        each = [_net_work(n, p, (), 1, True) for n, p in _pool(case["kind"], case["pool"], case["low"], case["high"])]
        parts = [(each[g], len(rows)) for g, rows in enumerate(members)]
    elif f == "serve":
        (net, path), pool = _serve_nets(case["pool"])
        parts = [(_net_work(net, path, (), 1, False), case["amplitudes"])]
        for j in range(case["partitions"]):
            parts.append((_net_work(*pool[j % case["pool"]], (), 1, True), 1))
    else:
        net, path, sliced = _network(_key(case))
        parts = [(_net_work(net, path, sliced, case.get("count", 1), _real(case)), 1)]
    return {"bytes": sum(w[0] * n for w, n in parts), "flops": sum(w[1] * n for w, n in parts)}


# ---- values in 64 bits ---------------------------------------------------------------------------

def _permuted(t, modes, order):
    """t (axes `modes`) with its axes in `order`; a flat gather for tensors of more axes than the strided copy kernels
    take."""
    if list(modes) == list(order):
        return t
    if len(modes) <= 12:
        return t.permute([modes.index(x) for x in order]).contiguous()
    stride, s = {}, 1
    for ax in range(len(modes) - 1, -1, -1):
        stride[modes[ax]] = s
        s *= t.shape[ax]
    left = torch.arange(t.numel(), device=t.device)
    at = torch.zeros_like(left)
    for x in reversed(order):
        e = t.shape[modes.index(x)]
        at += (left % e) * stride[x]
        left = left // e
    return t.reshape(-1)[at].reshape([t.shape[modes.index(x)] for x in order])


def _contract64(tensors, modes, pairs, open_modes, maxplus=False, batched=False):
    """The pairwise contraction of 64-bit torch tensors along a path; batched: a leading axis on every tensor."""
    live = [(t, list(m)) for t, m in zip(tensors, modes)]
    for i, j in pairs:
        (a, ma), (b, mb) = live[i], live[j]
        live[i] = live[j] = None
        K = [x for x in ma if x in mb]
        M, N = [x for x in ma if x not in K], [x for x in mb if x not in K]
        first = ["batch"] if batched else []
        lead = list(a.shape[:len(first)])
        size = lambda t, ms, of: [t.shape[len(first) + ms.index(x)] for x in of]
        sm, sn, sk = size(a, ma, M), size(b, mb, N), size(a, ma, K)
        a = _permuted(a, first + ma, first + M + K).reshape(lead + [math.prod(sm), math.prod(sk)])
        b = _permuted(b, first + mb, first + K + N).reshape(lead + [math.prod(sk), math.prod(sn)])
        if maxplus:
            c = a[..., :, 0:1] + b[..., 0:1, :]
            for q in range(1, a.shape[-1]):
                c = torch.maximum(c, a[..., :, q:q + 1] + b[..., q:q + 1, :])
        else:
            c = torch.matmul(a, b)
        live.append((c.reshape(lead + sm + sn), M + N))
    t, m = live[-1]
    return t if batched else _permuted(t, m, list(open_modes))


def exact(case, seed):
    f = case["family"]
    if f == "ensemble":
        pool = _pool(case["kind"], case["pool"], case["low"], case["high"])
        _, members = _ensemble_members(case)
        out = torch.zeros((case["count"], 2) if case["kind"] == "mis" else case["count"], dtype=torch.float64)
        for g, rows in enumerate(members):
            if len(rows) == 0:
                continue
            net, path = pool[g]
            # the leaves as handed over: rounded to FP32
            ts = [torch.tensor(t.astype(np.float32).astype(np.float64), device="cuda")
                  for t in _ensemble_leaves(case["kind"], net, seed * 64 + g, len(rows))]
            z = _contract64(ts, net.modes, path.pairs, (), case["kind"] == "mis", batched=True).cpu()
            if case["kind"] == "mis":
                out[rows, 0] = z
            else:
                out[rows] = torch.log(z)
        return out
    if f == "serve":
        (net, path), pool = _serve_nets(case["pool"])
        amps, lnz = [], []
        for i, leaves in _serve_requests(case, seed):
            n, p = (net, path) if i == 0 else pool[i - 1]
            ts = [torch.tensor(t.astype(np.complex128 if i == 0 else np.float64)) for t in leaves]
            v = _contract64(ts, n.modes, p.pairs, ())
            (amps if i == 0 else lnz).append(v.item() if i == 0 else math.log(v.item()))
        return {"amplitudes": np.array(amps, dtype=np.complex128), "ln_z": np.array(lnz)}
    net, path, sliced = _network(_key(case))
    if work(case)["flops"] > 1.2e13:  # at about 1 TFLOP/s in 64 bits
        return None
    ts = [t.to(torch.float64 if _real(case) else torch.complex128) for t in _inputs(case, seed)]
    if f == "mis":
        return _contract64(ts, net.modes, path.pairs, (), maxplus=True)
    total = 0.0
    for s in range(case.get("count", 1)):
        cut, at = {}, s
        for x in reversed(sliced):  # the first sliced label is the most significant digit
            cut[x], at = at % net.extent[x], at // net.extent[x]
        part = [t[tuple(cut.get(x, slice(None)) for x in m)] for t, m in zip(ts, net.modes)]
        total = total + _contract64(part, [[x for x in m if x not in cut] for m in net.modes], path.pairs,
                                    net.open_modes)
    if f == "spinglass":
        return torch.log(total).reshape(1)
    return total
