"""A server whose budget is a little below a plan's workspace: the request runs in the least memory that
its steps one by one take (no chains, no gate runs), with the same bits."""
import numpy as np
import pytest

from tests._lib import ensure_built
from tests.test_gate_run_lifetimes import gate_network
from tn_inputs import greedy, kicked_ising

pytestmark = pytest.mark.gpu


def state():
    return gate_network(17, 13, 2, seed=3)


def dynamics():
    net = kicked_ising.expectation_network(3, 7, 1.0, 0.9, 0.25, cols=3, lattice="square")
    return net, greedy.greedy_path(net, 3, 1.0, 0.0)


@pytest.mark.parametrize("make", [state, dynamics])
def test_budget_below_the_workspace(make):
    tn = ensure_built()
    net, path = make()
    plan = tn.Plan(net, path)
    steps = [plan.step(s) for s in range(len(path.pairs))]
    assert any(st["chain"] >= 0 or st["gate_run"] >= 0 for st in steps)
    ins = [np.ascontiguousarray(t, dtype=np.complex64) for t in net.tensors]
    want = np.zeros(plan.out_shape, dtype=np.complex128)
    plan.contract_host(ins, want)
    budget = plan.info()["workspace_bytes"] - 1
    srv = tn.Server(max_inflight=2, n_streams=2, hbm_budget_bytes=budget)
    tickets = [srv.submit(plan, ins) for _ in range(3)]
    for t in tickets:
        got = np.zeros_like(want)
        assert srv.poll(t, got) == tn.TN_OK, tn.last_error()
        assert got.tobytes() == want.tobytes()
    assert 0 < srv.stats()["hbm_in_use"] <= budget
    srv.destroy()
    plan.destroy()
