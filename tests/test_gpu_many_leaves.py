"""The staging launch's sizes: the leaves' addresses are parameters of the launch, up to 128, 512
and 3584 of them, and more leaves take more launches. Rings of n spins against the transfer
matrix's closed form: ln Z = n ln(2 cosh J) + ln(1 + tanh(J)^n); every one of the n steps and n
renormalised leaves rounds a few times at 2^-24."""
import numpy as np
import pytest
import torch

from tests._lib import ensure_built
from tn_inputs import ising_pf
from tn_inputs.network import Path

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [127, 128, 129, 512, 513, 3584, 3585])
def test_ring(n):
    tn = ensure_built()
    net = ising_pf.ring_network(n, 1.0, 1.0)
    cur, pairs = 0, []
    for i in range(1, n):
        pairs.append((cur, i))
        cur = n + i - 1
    plan = tn.Plan(net, Path(pairs), prec="r32_fp32", exp_scaling=True)
    inputs = [torch.tensor(np.ascontiguousarray(t, dtype=np.float32), device="cuda") for t in net.tensors]
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    log_scale = torch.zeros(1, dtype=torch.float64, device="cuda")
    for call in range(2):
        plan.contract(inputs, out, log_scale)
        got = float(torch.log(out) + log_scale)
        want = n * np.log(2 * np.cosh(1.0)) + np.log1p(np.tanh(1.0) ** n)
        assert abs(got - want) < 4 * n * 2.0 ** -23
    assert plan.launches_per_call() >= -(-n // 3584) + 1
