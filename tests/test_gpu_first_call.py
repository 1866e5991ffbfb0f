"""The first call of a new plan, on a non-blocking stream right after the plan was made: the tables that
the plan uploads have to be on the device by then, whatever stream the call is on."""
import numpy as np
import pytest
import torch

from tests._lib import ensure_built
from tn_inputs import greedy, kicked_ising, workloads

pytestmark = pytest.mark.gpu


def test_plan():
    tn = ensure_built()
    net = kicked_ising.expectation_network(3, 6, 1.0, 0.9, 0.25, cols=3, lattice="square")
    path = greedy.greedy_path(net, 3, 1.0, 0.0)
    ins = [torch.tensor(np.asarray(t), dtype=torch.complex64, device="cuda") for t in net.tensors]
    out = torch.zeros((), dtype=torch.complex128, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    got = []
    for _ in range(30):
        plan = tn.Plan(net, path)
        plan.contract(ins, out, stream=side)
        side.synchronize()
        got.append(complex(out.cpu()))
        plan.destroy()
    assert len(set(got)) == 1 and got[0] != 0


def test_batch():
    tn = ensure_built()
    ws = workloads.ising3r(64, seed=9)
    host = tn.Batch([w.net for w in ws], [w.path for w in ws], complex_=False, exp_scaling=True)
    packed = torch.tensor(host.pack([w.net for w in ws]), device="cuda")
    host.destroy()
    vals = torch.zeros((len(ws), 2), dtype=torch.float64, device="cuda")
    logs = torch.zeros(len(ws), dtype=torch.float64, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    first = None
    for _ in range(20):
        batch = tn.Batch([w.net for w in ws], [w.path for w in ws], complex_=False, exp_scaling=True)
        batch.contract(packed, vals, logs, stream=side)
        side.synchronize()
        now = torch.cat([vals[:, 0], logs]).clone()
        first = now if first is None else first
        assert torch.equal(now, first) and bool((vals[:, 0] > 0).all())
        batch.destroy()


def test_server():
    tn = ensure_built()
    w = workloads.random_circuit(3, 4, 8, 12)
    ins = [np.ascontiguousarray(t, dtype=np.complex64) for t in w.net.tensors]
    got = set()
    for _ in range(10):
        plan = tn.Plan(w.net, w.path)
        srv = tn.Server(max_inflight=2, n_streams=2)
        out = np.zeros((), dtype=np.complex128)
        assert srv.poll(srv.submit(plan, ins), out) == tn.TN_OK
        got.add(complex(out))
        srv.destroy()
        plan.destroy()
    assert len(got) == 1 and 0 not in got
