"""DARE's test for non-finite values sums four entries at a time, whatever the load's width: large
finite pseudo-gradients whose sums of four are finite are taken."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,values", [
    (torch.bfloat16, [6e37] * 8),                    # the sum of all eight of a load overflows
    (torch.float32, [3e38, -1e38, 3e38, -3e38]),     # as does a running sum, not that of the pairs
    (torch.bfloat16, [3e38, -1e38, 3e38, -3e38]),
])
def test_large_finite_values_are_taken(dtype, values):
    from paper_2607_03011_gb300 import isoloco as iso
    delta = torch.tensor(values * 16, device="cuda").to(dtype)
    N = delta.numel()
    plan = iso.Plan([(0, N, 0)], N, 1, dtype)
    theta, mom = torch.zeros(N, device="cuda"), torch.zeros(N, device="cuda")
    opts = iso.make_opts(outer_lr=0.5, momentum=0.0, sync=True, aggregator=2, sparsity=0.0)
    assert plan.diloco_outer_step(theta, mom, [-delta], opts) == 0
    assert torch.equal(mom, delta.float()) and torch.equal(theta, -0.5 * delta.float())


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("at", [0, 3, 5, 67])
def test_non_finite_values_are_reported(dtype, value, at):
    from paper_2607_03011_gb300 import isoloco as iso
    N = 68
    rep = torch.zeros(N, device="cuda", dtype=dtype)
    rep[at] = value
    plan = iso.Plan([(0, N, 0)], N, 1, dtype)
    theta, mom = torch.zeros(N, device="cuda"), torch.zeros(N, device="cuda")
    assert plan.diloco_outer_step(theta, mom, [rep], iso.make_opts(sync=True, aggregator=2, sparsity=0.9)) == iso.ERR_NONFINITE
