"""The launches a plan counts are the kernels that run (torch's profiler sees them)."""
import pytest
import torch

from paper_2607_03011_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MATS = [("a", 130, 65), ("b", 300, 257), ("v", 7, 0)]
GRAM_SIDE = [("s", 2100, 40)]
CALLS = [("ties", dict(aggregator=1, sparsity=0.3)), ("ties", dict(aggregator=1)), ("dare", dict(aggregator=2, sparsity=0.3)),
         ("mean", {})]


def kernels(run):
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]):  # the first use starts up slowly and may miss kernels
        run()
        torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        run()
        torch.cuda.synchronize()
    return sum("isoloco::" in e.name for e in prof.events())


def counted(plan, run):
    run()  # buffers of the first call
    seen = kernels(run)
    l0 = plan.launches
    run()
    return plan.launches - l0, seen


@pytest.mark.parametrize("K", [1, 8, 9, 17])
@pytest.mark.parametrize("kw", [kw for _, kw in CALLS], ids=[n for n, _ in CALLS])
def test_diloco_launches(K, kw):
    from paper_2607_03011_gb300 import isoloco as iso
    wl = W.make_workload(W.custom_spec(MATS, K=K, rank=2), seed=33, device="cuda")
    plan = iso.Plan(wl.table, wl.N, wl.K)
    th, b = wl.theta.clone(), wl.momentum.clone()
    n, seen = counted(plan, lambda: plan.diloco_outer_step(th, b, wl.replicas, iso.make_opts(sync=True, **kw)))
    assert n == seen


@pytest.mark.parametrize("shapes,kw", [(MATS, {}), (MATS + GRAM_SIDE, {}), (MATS, {"fast_steps": 5}), (MATS, {"spectrum_kind": 1}),
                                       (MATS, {"spectrum_kind": 3})])
def test_outer_step_launches(shapes, kw):
    from paper_2607_03011_gb300 import isoloco as iso
    wl = W.make_workload(W.custom_spec(shapes, K=2, rank=2, momentum_std=1e-4), seed=34, device="cuda")
    plan = iso.Plan(wl.table, wl.N, wl.K)
    th, b = wl.theta.clone(), wl.momentum.clone()

    def run():
        th.copy_(wl.theta)
        b.copy_(wl.momentum)
        assert plan.outer_step(th, b, wl.replicas, iso.make_opts(sync=True, **kw)) == 0

    n, seen = counted(plan, run)
    assert n == seen
