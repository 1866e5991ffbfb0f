"""Gate chains with a launch per step: the leaf's tiled permutation, the streaming kernel in every form (k = 2 from
registers, k = 4, 8, 16 by bulk copies) and the widening, which a chain without scaling and slices only
reaches when its output overlaps the leaf. The profile shows that these kernels ran."""
import numpy as np
import pytest
import torch

import oracle
from tests._lib import ensure_built
from tests.test_gpu_parity import gate_chain_network
from tn_inputs import circuits

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tn():
    return ensure_built()


def overlapping(tensors, out_elems, real):
    """(leaves, output): the state at the start of a buffer, the output from its last elements on."""
    leaf, final, size = (torch.float32, torch.float64, 4) if real else (torch.complex64, torch.complex128, 8)
    n = tensors[0].numel()
    buf = torch.zeros((n - 4) * size + out_elems * 2 * size, dtype=torch.uint8, device="cuda")
    state = buf[:n * size].view(leaf)
    state.copy_(tensors[0].reshape(-1))
    return [state] + tensors[1:], buf[(n - 4) * size:].view(final)


def contract(tn, plan, leaves, out, gates, state_bytes, log_scale=None):
    """The call, with as many streaming launches as gates and the whole state staged (read and written)."""
    plan.profile(True)
    plan.contract(leaves, out, log_scale)
    prof = plan.profile_read()
    plan.profile(False)
    assert prof["launches"][tn.TN_CLASS_STREAM] == gates
    assert prof["bytes"][4] >= 2 * state_bytes


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("arity", [1, 2, 3, 4])
def test_stream_forms(tn, arity, real):
    """m = 2^18 / k rows: 2^14 and more, so k = 4, 8, 16 take the bulk-copy form (8192 rows or more). Bound:
    per gate of depth k, 2 k roundings a component, times the 2-norm of |U| (at most sqrt(k)) and sqrt(2)
    for the components, and 2 more for the gate's and the state's entries, in the 2-norm."""
    gates, k = 5, 2 ** arity
    net, path = gate_chain_network(n_qubits=18, n_gates=gates, seed=40 + arity, arity=arity, real=real)
    plan = tn.Plan(net, path, prec="r32_fp32" if real else "fp32")
    steps = [plan.step(s) for s in range(gates)]
    assert all(st["cls"] == tn.TN_CLASS_STREAM and st["k"] == k and st["m"] >= 8192 for st in steps)
    tensors = [torch.tensor(np.asarray(t)).to(torch.float32 if real else torch.complex64).cuda() for t in net.tensors]
    leaves, out = overlapping(tensors, 1 << 18, real)
    contract(tn, plan, leaves, out, gates, (4 if real else 8) << 18)
    plan.destroy()
    want = oracle.contract(net, path).reshape(-1)
    bound = gates * (2 * k * np.sqrt(k) * np.sqrt(2) + 2) * 2.0 ** -24
    assert np.linalg.norm(out.cpu().numpy() - want) <= bound * np.linalg.norm(want)


@pytest.mark.parametrize("arity", [1, 2, 3, 4])
def test_stream_forms_scaled(tn, arity):
    """The same with exponent scaling (a launch per step whatever the buffers): operands read through their
    powers of two, so the bits times the log scale are those without it."""
    net, path = gate_chain_network(n_qubits=18, n_gates=4, seed=50 + arity, arity=arity)
    tensors = [torch.tensor(np.asarray(t)).to(torch.complex64).cuda() for t in net.tensors]
    out = [torch.zeros(1 << 18, dtype=torch.complex128, device="cuda") for _ in range(2)]
    log_scale = torch.zeros(1, dtype=torch.float64, device="cuda")
    plan = tn.Plan(net, path)
    plan.contract(tensors, out[0])
    plan.destroy()
    plan = tn.Plan(net, path, exp_scaling=True)
    assert all(plan.step(s)["gate_run"] == -1 for s in range(4))
    contract(tn, plan, tensors, out[1], 4, 8 << 18, log_scale)
    plan.destroy()
    back = 2.0 ** round(log_scale.item() / np.log(2.0))
    assert abs(np.log(back) - log_scale.item()) < 1e-12
    assert torch.equal(torch.view_as_real(out[1] * back), torch.view_as_real(out[0]))


@pytest.mark.parametrize("qubits,seed", [(20, 1), (23, 2), (26, 26)])
def test_permuted_state(tn, qubits, seed):
    """A state in a shuffled declared order, staged by the permutation kernel, against the run that reads it in
    place (which is checked against the oracle elsewhere): the same bits."""
    net = circuits.state_network(qubits, 3, seed)
    path = circuits.state_path(net)
    plan = tn.Plan(net, path)
    assert plan.tensor(0)["tiled"] >= 1 and plan.step(0)["gate_run"] == 0
    tensors = [torch.tensor(np.asarray(t), dtype=torch.complex64, device="cuda") for t in net.tensors]
    want = torch.zeros(1 << qubits, dtype=torch.complex128, device="cuda")
    plan.contract(tensors, want)
    leaves, out = overlapping(tensors, 1 << qubits, False)
    contract(tn, plan, leaves, out, 3, 8 << qubits)
    plan.destroy()
    assert torch.equal(torch.view_as_real(out).view(torch.int64), torch.view_as_real(want).view(torch.int64))


@pytest.mark.parametrize("arity", [1, 4])
def test_a_single_gate_is_not_slower_in_a_run(tn, arity):
    """One gate on a real 26-qubit state: the run (which saves the staging and the widening) against the launch
    per step of a call whose output overlaps the leaf, the best of several calls each."""
    net, path = gate_chain_network(n_qubits=26, n_gates=1, seed=60 + arity, arity=arity, real=True)
    plan = tn.Plan(net, path, prec="r32_fp32")
    assert plan.step(0)["gate_run"] == 0
    tensors = [torch.tensor(np.asarray(t)).to(torch.float32).cuda() for t in net.tensors]
    out = torch.zeros(1 << 26, dtype=torch.float64, device="cuda")
    leaves, over = overlapping(tensors, 1 << 26, True)

    def best(ins, o):
        times = []
        for _ in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            leaves[0].copy_(tensors[0].reshape(-1))
            e0.record()
            plan.contract(ins, o)
            e1.record()
            torch.cuda.synchronize()
            times.append(e0.elapsed_time(e1))
        return min(times)

    run, steps = best(tensors, out), best(leaves, over)
    plan.destroy()
    assert run < steps
