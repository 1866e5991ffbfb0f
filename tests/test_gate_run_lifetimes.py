"""Gate runs on the plan's own offsets: a run executes in one launch, so its output is written while
its input and its gates are still read, by thread blocks in any order. A CPU replay of host-only plans
executes each run as one event in its worst order, every store before any load: what a run reads
from memory that it writes comes back as NaN. A leaf that a run reads where the caller has it, and the
output of a run that ends the path, are not in the workspace. Inner results of a run are never stored."""
import numpy as np
import pytest

import oracle
from tests._lib import ensure_built
from tests.test_plan_emulator import offsets
from tn_inputs import greedy, kicked_ising
from tn_inputs.network import Network, Path


@pytest.fixture(scope="module")
def tn():
    return ensure_built()


def gate_network(qubits, gates, arity, where="first", project=0, seed=0, real=False):
    """A state of `qubits` qubits declared before, between or after its gates; `project` qubits are
    then contracted with vectors, one after another."""
    rng = np.random.default_rng(seed)
    noise = lambda *shape: rng.standard_normal(shape) + (0.0 if real else 1j * rng.standard_normal(shape))
    wire, label = list(range(qubits)), qubits
    tensors, modes = [], []
    for _ in range(gates):
        qs = [int(q) for q in rng.choice(qubits, size=arity, replace=False)]
        new = list(range(label, label + arity))
        tensors.append(np.linalg.qr(noise(2 ** arity, 2 ** arity))[0].reshape((2,) * (2 * arity)))
        modes.append(tuple(new) + tuple(wire[q] for q in qs))
        for q, x in zip(qs, new):
            wire[q] = x
        label += arity
    for q in range(project):
        tensors.append(noise(2))
        modes.append((wire[q],))
    at = {"first": 0, "between": gates // 2, "last": len(tensors)}[where]
    tensors.insert(at, noise(*(2,) * qubits))
    modes.insert(at, tuple(range(qubits)))
    net = Network(tensors, modes, {x: 2 for x in range(label)}, tuple(wire[project:]))
    net.check()
    pairs, cur, T = [], at, len(tensors)
    for g in [i for i in range(T) if i != at]:
        pairs.append((cur, g))
        cur = T + len(pairs) - 1
    return net, Path(pairs)


def runs_of(steps):
    """{first step: steps of the run}."""
    out = {}
    for s, st in enumerate(steps):
        if st["gate_run"] >= 0:
            first = next(q for q in range(s + 1) if steps[q]["gate_run"] == st["gate_run"])
            out.setdefault(first, []).append(s)
    return out


def replay_runs(plan, net, real):
    info, planes = plan.info(), 1 if real else 2
    T, S = net.n_tensors, info["n_steps"]
    ws = np.full(info["workspace_bytes"] // 4 + 1, np.nan)
    tens = [plan.tensor(t) for t in range(T + S)]
    steps = [plan.step(s) for s in range(S)]
    runs = runs_of(steps)

    def where(t):
        return slice(tens[t]["offset"] // 4, tens[t]["offset"] // 4 + planes * tens[t]["size"])

    def read(t):
        v = ws[where(t)].reshape(planes, -1)
        return v[0].copy() if real else v[0] + 1j * v[1]

    def write(t, v):
        ws[where(t)] = v if real else np.concatenate([v.real, v.imag])

    def declared(t):
        a = np.asarray(net.tensors[t])
        return np.transpose(a, [net.modes[t].index(x) for x in plan.layout(t)]).ravel()

    def product(st, a, b):
        out = np.empty(st["m"] * st["n"], dtype=np.result_type(a, b))
        idx = offsets(st["rows"], st["m"])[:, None] + offsets(st["cols"], st["n"])[None, :]
        out[idx] = a.reshape(st["m"], st["k"]) @ b.reshape(st["n"], st["k"]).T
        return out

    for t in range(T):
        write(t, declared(t))
    root, s = None, 0
    while s < S:
        group = runs.get(s, [s])
        st, last = steps[s], group[-1]
        direct = s in runs and st["a_id"] < T  # (every leaf here has power-of-two extents and no slices)
        if s in runs and last < S - 1:
            ws[where(T + last)] = np.nan
        x = declared(st["a_id"]) if direct else read(st["a_id"])
        for q in group:
            x = product(steps[q], x, read(steps[q]["b_id"]))
        if last < S - 1:
            write(T + last, x)
        else:
            root = x
        s = last + 1
    return root.reshape(tuple(net.extent[x] for x in net.open_modes)), runs


def check(tn, net, path, prec, real=False, runs_at_least=1):
    plan = tn.Plan(net, path, prec=prec, host_only=True)
    got, runs = replay_runs(plan, net, real)
    plan.destroy()
    assert len(runs) >= runs_at_least
    want = oracle.contract(net, path)
    assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()


@pytest.mark.parametrize("where", ["first", "between", "last"])
@pytest.mark.parametrize("project", [0, 5])
@pytest.mark.parametrize("qubits,gates,arity", [(16, 20, 2), (16, 16, 3), (17, 2, 2), (18, 14, 2), (15, 24, 1)])
def test_states(tn, qubits, gates, arity, where, project):
    # gates of one pair of wires in a row may take few runs: only longer lists must have several
    net, path = gate_network(qubits, gates, arity, where, project, seed=qubits * gates + project)
    check(tn, net, path, "fp32", runs_at_least=2 if gates >= 14 and arity > 1 else 1)


@pytest.mark.parametrize("seed", range(4))
def test_real_states(tn, seed):
    net, path = gate_network(16, 18, 2, ("first", "last")[seed % 2], 3 * (seed // 2), seed=seed, real=True)
    check(tn, net, path, "r32_fp32", real=True, runs_at_least=2)


@pytest.mark.parametrize("rows,cols,steps,seed,alpha,prec", [(4, 4, 6, 43, 0.5, "3xtf32"), (4, 3, 11, 14, 0.5, "fp32"),
                                                             (4, 3, 11, 14, 1.0, "fp32")])
def test_kicked_ising(tn, rows, cols, steps, seed, alpha, prec):
    net = kicked_ising.expectation_network(rows, steps, 1.0, 0.9, 0.25, cols=cols, lattice="square")
    path = greedy.greedy_path(net, seed, alpha, 0.0)
    check(tn, net, path, prec, runs_at_least=0)
