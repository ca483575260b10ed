"""A step whose cooperative launch of the polar loop is refused runs its iterations as ordinary
launches (faked on the host: the launch is not made), with the loop's bits."""
import pytest
import torch

from paper_2607_03011_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [("a", 130, 65), ("b", 65, 130), ("c", 257, 257), ("d", 300, 520), ("v", 7, 0)]
GRAM_SIDE = [("s", 2100, 40)]  # (with full precision it would keep the plan off the loop)


@pytest.mark.parametrize("kw,shapes", [({}, SHAPES + GRAM_SIDE), ({"full_precision": 1}, SHAPES),
                                       ({"fast_steps": 5}, SHAPES), ({"spectrum_kind": 1}, SHAPES)])
def test_refused_loop_falls_back(kw, shapes):
    from paper_2607_03011_gb300 import isoloco as iso
    wl = W.make_workload(W.custom_spec(shapes, K=2, rank=2, momentum_std=1e-4), seed=31, device="cuda")
    plan = iso.Plan(wl.table, wl.N, wl.K)

    def step():
        th, b, upd = wl.theta.clone(), wl.momentum.clone(), torch.empty_like(wl.theta)
        l0 = plan.launches
        assert plan.outer_step(th, b, wl.replicas, iso.make_opts(1.0, 0.7, 0.9, sync=True, **kw), update_out=upd) == 0
        return th, b, upd, plan.launches - l0

    want = step()
    assert iso.lib().isoloco_debug_refuse_loop(plan._h, 1) == 0
    got, again = step(), step()
    for w, g, a in zip(want[:3], got, again):
        assert torch.equal(w, g) and torch.equal(w, a)
    assert got[3] > want[3] + 10 and again[3] == want[3]
