"""Profiling with single launches: every phase of every polar iteration is a launch of its own,
with the bits of the loop's kernel (or of the graph, where a plan does not take the loop)."""
import pytest
import torch

from paper_2607_03011_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LOOP = [("a", 130, 65), ("b", 65, 130), ("c", 257, 257), ("s", 2100, 40), ("v", 7, 0)]
SPLIT_GRAM = [("a", 4200, 600), ("b", 300, 257)]  # 600 columns: not Gram-side


@pytest.mark.parametrize("shapes,kw", [(LOOP, {}), (SPLIT_GRAM, {}), (LOOP, {"spectrum_kind": 2})])
def test_profile_with_single_launches(shapes, kw):
    from paper_2607_03011_gb300 import isoloco as iso
    wl = W.make_workload(W.custom_spec(shapes, K=2, rank=2, momentum_std=1e-4), seed=32, device="cuda")
    plan = iso.Plan(wl.table, wl.N, wl.K)

    def step():
        th, b, upd = wl.theta.clone(), wl.momentum.clone(), torch.empty_like(wl.theta)
        l0 = plan.launches
        assert plan.outer_step(th, b, wl.replicas, iso.make_opts(1.0, 0.7, 0.9, sync=True, **kw), update_out=upd) == 0
        return th, b, upd, plan.launches - l0

    want = step()
    plan.profile(2)
    got = step()
    phases = plan.profile_read()
    plan.profile(False)
    again = step()
    for w, g, a in zip(want[:3], got, again):
        assert torch.equal(w, g) and torch.equal(w, a)
    iters = max(plan.read_diag()["iters"])
    for name in ("gram", "control", "poly", "update"):
        ms, n = phases[name]
        assert n >= iters and ms > 0.0, (name, phases[name], iters)
    assert again[3] == want[3]
