"""Step chains run by tree level: the workspace offsets have to hold for that order too. A CPU
replay of plans on their own offsets, every chain's steps executed level by level with a level's
results written only after all of its operands were read and in reverse order, over several
passes, against the oracle; and on the GPU, networks of odd extents with wide and deep chains."""
import numpy as np
import pytest

import oracle
from tests._lib import ensure_built
from tests.test_plan_emulator import offsets
from tests.test_oracle_pins import random_network
from tn_inputs import greedy, workloads


def execution_order(steps, T):
    """[[steps run together], ...]: single steps, and the levels of each chain."""
    out, s = [], 0
    while s < len(steps):
        if steps[s]["chain"] < 0:
            out.append([s])
            s += 1
            continue
        e = s
        while e < len(steps) and steps[e]["chain"] == steps[s]["chain"]:
            e += 1
        level = {}
        for q in range(s, e):
            ops = [steps[q][x] - T for x in ("a_id", "b_id")]
            level[q] = max([level[o] + 1 for o in ops if o >= s], default=0)
        for lv in range(max(level.values()) + 1):
            out.append([q for q in reversed(range(s, e)) if level[q] == lv])
        s = e
    return out


def replay_levels(plan, net, sliced):
    info = plan.info()
    T, S, B, n = net.n_tensors, info["n_steps"], info["slice_batch"], info["n_slices"]
    ws = np.full(info["workspace_bytes"] // 4 + 1, np.nan)
    tens = [plan.tensor(t) for t in range(T + S)]
    steps = [plan.step(s) for s in range(S)]
    copy = lambda t, b: tens[t]["offset"] // 4 + 2 * (b if tens[t]["batched"] else 0) * tens[t]["size"]

    def read(t, b):
        at, z = copy(t, b), tens[t]["size"]
        return ws[at: at + z] + 1j * ws[at + z: at + 2 * z]

    total = 0.0
    for p in range(-(-n // B)):
        nb = min(B, n - p * B)
        for t in range(T):
            if p > 0 and not tens[t]["batched"]:
                continue
            for b in range(nb if tens[t]["batched"] else 1):
                sid, vals = p * B + b, {}
                for x in reversed(sliced):
                    vals[x], sid = sid % net.extent[x], sid // net.extent[x]
                a = np.asarray(net.tensors[t])[tuple(vals.get(x, slice(None)) for x in net.modes[t])]
                kept = [x for x in net.modes[t] if x not in vals]
                a = np.transpose(a, [kept.index(x) for x in plan.layout(t)]).ravel()
                at = copy(t, b)
                ws[at: at + a.size], ws[at + a.size: at + 2 * a.size] = a.real, a.imag
        for group in execution_order(steps, T):
            made = []
            for s in group:
                st = steps[s]
                if p > 0 and not st["batched"]:
                    continue
                for b in range(nb if st["batched"] else 1):
                    c = read(st["a_id"], b).reshape(st["m"], st["k"]) @ read(st["b_id"], b).reshape(st["n"], st["k"]).T
                    made.append((s, b, c))
            for s, b, c in made:
                st, at = steps[s], copy(T + s, b)
                idx = offsets(st["rows"], st["m"])[:, None] + offsets(st["cols"], st["n"])[None, :]
                ws[at + idx], ws[at + tens[T + s]["size"] + idx] = c.real, c.imag
        root = T + S - 1
        for b in range(nb if tens[root]["batched"] else 1):
            total = total + read(root, b)
    return np.asarray(total).reshape(tuple(net.extent[x] for x in net.open_modes))


@pytest.mark.parametrize("batch", [1, 3, 16])
def test_level_order_fits_the_offsets(batch):
    tn = ensure_built()
    w = workloads.random_circuit(3, 4, 8, 3, n_sliced=4)
    plan = tn.Plan(w.net, w.path, w.sliced, max_slice_batch=batch, host_only=True)
    steps = [plan.step(s) for s in range(len(w.path.pairs))]
    assert len(execution_order(steps, w.net.n_tensors)) < len(steps)
    got = replay_levels(plan, w.net, w.sliced)
    plan.destroy()
    want = oracle.contract(w.net, w.path, w.sliced)
    assert abs(got - want) < 1e-12 * abs(want)


@pytest.mark.gpu
@pytest.mark.parametrize("seed", range(6))
@pytest.mark.parametrize("real", [False, True])
def test_chains_of_odd_extents(seed, real):
    """Random networks, extents 2 and 3 (no shifts in the offset maps), open labels: one chain for
    the whole path. A-priori bound: each step of depth k adds at most 2 (2 k + 2) 2^-24 and each
    leaf's rounding 2^-24, relative to the contraction of the absolute values."""
    tn = ensure_built()
    net = random_network(900 + seed, n_tensors=14, n_labels=24, n_open=2)
    if real:
        net.tensors = [np.abs(np.asarray(t)) for t in net.tensors]
    path = greedy.greedy_path(net, seed=seed)
    plan = tn.Plan(net, path, prec="r32_fp32" if real else "fp32", exp_scaling=real)
    dt = np.float32 if real else np.complex64
    host = [np.ascontiguousarray(t, dtype=dt) for t in net.tensors]
    out, ls = np.zeros(plan.out_shape, dtype=np.float64 if real else np.complex128), np.zeros(1)
    plan.contract_host(host, out, ls)
    chained = sum(plan.step(s)["chain"] >= 0 for s in range(len(path.pairs)))
    depths = [plan.step(s)["k"] for s in range(len(path.pairs))]
    plan.destroy()
    assert chained > 0
    want = oracle.contract(net, path)
    net.tensors = [np.abs(np.asarray(t)) for t in net.tensors]
    terms = sum(2 * (2 * k + 2) for k in depths) + net.n_tensors
    assert np.all(np.abs(out * np.exp(ls[0]) - want) <= terms * 2.0 ** -24 * oracle.contract(net, path))
