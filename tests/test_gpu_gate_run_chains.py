"""Several gate runs one after another (a run from an intermediate to an intermediate among them), against
the general path bit for bit, against repeated calls, the graph and the host form, and against the
oracle. A call whose output overlaps the leaf that the first run reads takes the general path."""
import numpy as np
import pytest
import torch

import oracle
from tests._lib import FP32_BAR, ensure_built
from tests.test_gate_run_lifetimes import gate_network
from tn_inputs import greedy, kicked_ising

pytestmark = pytest.mark.gpu


def bits(x):
    return torch.view_as_real(x).view(torch.int64) if x.is_complex() else x.view(torch.int64)


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("qubits,gates,arity,where,project", [(16, 20, 2, "first", 0), (16, 16, 3, "between", 0),
                                                              (17, 14, 2, "last", 5), (18, 14, 2, "between", 3),
                                                              (20, 24, 2, "last", 0), (24, 16, 2, "first", 0)])
def test_same_bits_as_a_pass_per_step(real, qubits, gates, arity, where, project):
    tn = ensure_built()
    net, path = gate_network(qubits, gates, arity, where, project, seed=qubits + gates, real=real)
    plan = tn.Plan(net, path, prec="r32_fp32" if real else "fp32")
    assert max(plan.step(s)["gate_run"] for s in range(gates)) >= 1
    leaf, final = (torch.float32, torch.float64) if real else (torch.complex64, torch.complex128)
    tensors = [torch.tensor(np.asarray(t)).to(leaf).cuda() for t in net.tensors]
    state = max(range(len(tensors)), key=lambda t: tensors[t].numel())
    out = torch.zeros(1 << (qubits - project), dtype=final, device="cuda")
    first = None
    for _ in range(3):
        plan.contract(tensors, out)
        first = bits(out).clone() if first is None else first
        assert torch.equal(bits(out), first)
    for _ in range(2):
        out.zero_()
        plan.contract_graph(tensors, out)
        assert torch.equal(bits(out), first)
    host = np.zeros(plan.out_shape, dtype=np.float64 if real else np.complex128)
    plan.contract_host([np.ascontiguousarray(t.cpu().numpy()) for t in tensors], host)
    assert torch.equal(bits(torch.tensor(host).reshape(-1)), first.cpu())
    size = 4 if real else 8
    n = tensors[state].numel()
    buf = torch.zeros(3 * n * size, dtype=torch.uint8, device="cuda")
    over = list(tensors)
    over[state] = buf[:n * size].view(leaf)
    over[state].copy_(tensors[state].reshape(-1))
    at = (n - 4) * size
    out2 = buf[at:at + out.numel() * 2 * size].view(final)
    plan.contract(over, out2)
    assert torch.equal(bits(out2), first)
    plan.destroy()
    if project == 0:
        # per gate of depth k = 2^arity: 2 k roundings a component, times the 2-norm of |U| (at most
        # sqrt(k)) and sqrt(2) for the components; 2 more for the gate's and the state's entries
        k = 2 ** arity
        bound = gates * (2 * k * np.sqrt(k) * np.sqrt(2) + 2) * 2.0 ** -24
        want = oracle.contract(net, path).reshape(-1)
        assert np.linalg.norm(out.cpu().numpy() - want) <= bound * np.linalg.norm(want)


def test_kicked_ising():
    tn = ensure_built()
    net = kicked_ising.expectation_network(4, 6, 1.0, 0.9, 0.25, cols=4, lattice="square")
    path = greedy.greedy_path(net, 43, 0.5, 0.0)
    plan = tn.Plan(net, path, prec="3xtf32")
    runs = [plan.step(s)["gate_run"] for s in range(len(path.pairs))]
    assert max(runs) >= 0
    host = [np.ascontiguousarray(t, dtype=np.complex64) for t in net.tensors]
    got = []
    for _ in range(4):
        out = np.zeros((), dtype=np.complex128)
        plan.contract_host(host, out)
        got.append(complex(out))
    plan.destroy()
    assert len(set(got)) == 1
    assert abs(got[0] - oracle.contract(net, path)) < FP32_BAR


def test_log_scale_in_the_leaf():
    """The log scale (0 without scaling) in the memory of the leaf that the run reads: the general path, with
    the bits of separate buffers."""
    tn = ensure_built()
    net, path = gate_network(18, 4, 2, seed=5)
    plan = tn.Plan(net, path)
    tensors = [torch.tensor(np.asarray(t)).to(torch.complex64).cuda() for t in net.tensors]
    out = torch.zeros(1 << 18, dtype=torch.complex128, device="cuda")
    plan.contract(tensors, out)
    want = bits(out).clone()
    plan.profile(True)
    plan.contract(tensors, out)
    assert plan.profile_read()["launches"][tn.TN_CLASS_STREAM] == 1
    inside = tensors[0].reshape(-1)[1000:1001].view(torch.float64)
    plan.contract(tensors, out, inside)
    assert plan.profile_read()["launches"][tn.TN_CLASS_STREAM] == 4
    assert torch.equal(bits(out), want) and inside.item() == 0.0
    plan.destroy()
