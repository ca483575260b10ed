"""The reduction and apply passes where 16-byte vectors do not fit: matrices whose rows are
padded in the planes, or that start off a 16-byte boundary."""
import pytest
import torch

from paper_2607_03011_gb300 import workloads as W
from parity import check_step, oracle_step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def iso():
    from paper_2607_03011_gb300 import isoloco
    isoloco.lib()
    return isoloco


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("K", [1, 4, 5, 9])
@pytest.mark.parametrize("pmode", [0, 1])
def test_same_bits_on_and_off_a_16_byte_boundary(iso, dtype, K, pmode):
    """Matrices with whole rows of vectors, moved by one element by a scalar parameter."""
    spec = W.custom_spec([("a", 64, 512), ("b", 1000, 8), ("c", 8, 1032)], K=K, rank=2, momentum_std=1e-4,
                         replica_dtype=dtype)
    wl = W.make_workload(spec, seed=5, device="cuda")
    opts = iso.make_opts(1.0, 0.7, 0.9, sync=True, **({"orth_target": pmode} if pmode else {}))

    def step(table, theta, mom, reps):
        theta, mom, upd = theta.clone(), mom.clone(), torch.empty_like(theta)
        plan = iso.Plan(table, theta.numel(), K, reps[0].dtype)
        assert plan.outer_step(theta, mom, reps, opts, update_out=upd) == 0
        return theta, mom, upd

    want = step(wl.table, wl.theta, wl.momentum, list(wl.replicas))
    moved = [(0, 1, 0)] + [(o + 1, r, c) for o, r, c in wl.table]
    one = torch.ones(1, device="cuda")
    got = step(moved, torch.cat([one, wl.theta]), torch.cat([one, wl.momentum]),
               [torch.cat([one.to(r.dtype), r]) for r in wl.replicas])
    for w, g in zip(want, got):
        assert torch.equal(w, g[1:])


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("shapes", [
    [("p", 3, 0), ("a", 5, 1), ("b", 1, 5), ("c", 259, 255)],
    [("a", 3, 32767), ("b", 3, 32768), ("c", 2, 65537)],   # either side of the longest row divided by multiplication
    [("a", 70001, 1), ("p", 1, 0), ("b", 30001, 3)],
])
def test_padded_rows_match_oracle(iso, shapes, dtype):
    spec = W.custom_spec(shapes, K=3, rank=1, momentum_std=1e-4, replica_dtype=dtype)
    wl = W.make_workload(spec, seed=6, device="cuda")
    plan = iso.Plan(wl.table, wl.N, wl.K, wl.replicas[0].dtype)
    th, b, upd = wl.theta.clone(), wl.momentum.clone(), torch.empty_like(wl.theta)
    assert plan.outer_step(th, b, wl.replicas, iso.make_opts(1.0, 0.7, 0.9, sync=True), update_out=upd) == 0
    ref = oracle_step(wl.table, wl.theta, wl.momentum, wl.replicas, 1.0, 0.7, 0.9)
    ref["theta_in"] = wl.theta.double().cpu().numpy()
    check_step(wl.table, th.double().cpu().numpy(), b.double().cpu().numpy(), upd.double().cpu().numpy(),
               plan.read_diag()["sigma_bar"], ref)
