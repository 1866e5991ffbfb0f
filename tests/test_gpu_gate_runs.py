"""Gate runs against the general path (staging, a pass per step, widening), bit for bit. A call whose
output overlaps the state's leaf takes the general path, since a run writes the output while it reads
the leaf: so each network is contracted once with separate buffers and once with buffers that
overlap by two elements. Every gate size, runs split by the tile's size, runs of one step, and tiles
of 2^8 to 2^13 elements; the oracle checks the values."""
import numpy as np
import pytest
import torch

import oracle
from tests._lib import ensure_built
from tests.test_gpu_parity import gate_chain_network

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("qubits,gates,arity", [(11, 1, 1), (12, 2, 2), (12, 5, 2), (13, 3, 3), (14, 2, 4), (14, 9, 2),
                                                (15, 6, 3), (16, 4, 2), (16, 12, 1), (18, 9, 2), (19, 4, 4), (20, 4, 2)])
def test_same_bits_as_a_pass_per_step(real, qubits, gates, arity):
    tn = ensure_built()
    net, path = gate_chain_network(n_qubits=qubits, n_gates=gates, seed=qubits + gates, arity=arity, real=real)
    plan = tn.Plan(net, path, prec=tn.TN_R32_FP32_SIMT if real else 0)
    assert all(plan.step(s)["cls"] == tn.TN_CLASS_STREAM for s in range(gates))
    few = plan.launches_per_call()
    assert few <= 2 + gates  # staging, runs (or steps), at most one more
    leaf, final = (torch.float32, torch.float64) if real else (torch.complex64, torch.complex128)
    tensors = [torch.tensor(np.asarray(t)).to(leaf).cuda() for t in net.tensors]
    n, size = 1 << qubits, 4 if real else 8
    out = torch.zeros(n, dtype=final, device="cuda")
    log_scale = torch.full((1,), 7.0, dtype=torch.float64, device="cuda")
    plan.contract(tensors, out, log_scale)
    assert log_scale.item() == 0.0
    buf = torch.zeros(3 * n * size, dtype=torch.uint8, device="cuda")
    state = buf[:n * size].view(leaf)
    state.copy_(tensors[0].reshape(-1))
    over = buf[(n - 4) * size:(n - 4) * size + 2 * n * size].view(final)
    plan.contract([state] + tensors[1:], over)
    assert torch.equal(out.view(torch.int64) if real else torch.view_as_real(out).view(torch.int64),
                       over.view(torch.int64) if real else torch.view_as_real(over).view(torch.int64))
    want = oracle.contract(net, path).reshape(-1)
    assert np.abs(out.cpu().numpy() - want).max() / np.abs(want).max() < 1e-5
