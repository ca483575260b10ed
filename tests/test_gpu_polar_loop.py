"""The polar loop (one persistent kernel for iterations 1, 2, ...) at the sizes where its walk
over the tiles can go wrong, against the fp64 oracle and, bit for bit, against the same step
with its iterations as single launches (a stream capture takes that path)."""
import pytest
import torch

from paper_2607_03011_gb300 import workloads as W
from parity import check_step, oracle_step

pytestmark = pytest.mark.gpu

SETS = {
    "one tile": [("a", 64, 64)],
    "tile edges": [("a", 255, 255), ("b", 256, 256), ("c", 257, 257), ("d", 256, 513), ("e", 513, 256)],
    "columns split between the epilogue's halves": [("a", 33, 33), ("b", 65, 65), ("c", 97, 97), ("d", 129, 129),
                                                    ("e", 160, 193), ("f", 290, 64), ("g", 64, 290), ("h", 300, 320)],
    "tiles read transposed": [("a", 513, 514), ("b", 600, 1100), ("c", 1100, 600), ("d", 2600, 300), ("e", 769, 1793)],
    "more matrices than a warp has lanes": [(f"a{i}", 24, 40) for i in range(37)] + [(f"b{i}", 40, 24) for i in range(3)],
    "Gram side beside others": [(f"a{i}", 2048, 16) for i in range(3)] + [("b", 300, 200), ("c", 520, 65)],
    "more groups than the small parameters hold": [(f"a{i}", 20 + i, 33) for i in range(13)],
    "more groups than the parameters hold (graph of launches)": [(f"a{i}", 30 + i, 33) for i in range(40)],
}


@pytest.fixture(scope="module")
def iso():
    from paper_2607_03011_gb300 import isoloco
    isoloco.lib()
    return isoloco


def captured_step(plan, iso, wl):
    """The step with its iterations as single launches."""
    th, b, upd = wl.theta.clone(), wl.momentum.clone(), torch.empty_like(wl.theta)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.outer_step(th, b, wl.replicas, iso.make_opts(1.0, 0.7, 0.9), update_out=upd)
    graph.replay()
    torch.cuda.synchronize()
    return th, b, upd


@pytest.mark.parametrize("count", [60, 76])  # Gram's tiles about the eight waves from which phases alternate
def test_walk_in_both_directions(iso, count):
    """Enough tiles that the phases walk in opposite directions, with Gram-side matrices beside."""
    shapes = [(f"a{i}", 1000, 1021) for i in range(count)] + [("s0", 4100, 500), ("s1", 4100, 500)]
    wl = W.make_workload(W.custom_spec(shapes, K=1, rank=2, momentum_std=1e-4), seed=24, device="cuda")
    plan = iso.Plan(wl.table, wl.N, wl.K)
    th, b, upd = wl.theta.clone(), wl.momentum.clone(), torch.empty_like(wl.theta)
    assert plan.outer_step(th, b, wl.replicas, iso.make_opts(1.0, 0.7, 0.9, sync=True), update_out=upd) == 0
    for got, want in zip((th, b, upd), captured_step(plan, iso, wl)):
        assert torch.equal(got, want)


@pytest.mark.parametrize("name", list(SETS))
def test_loop_matches_oracle_and_single_launches(iso, name):
    spec = W.custom_spec(SETS[name], K=2, rank=2, momentum_std=1e-4)
    wl = W.make_workload(spec, seed=23, device="cuda")
    plan = iso.Plan(wl.table, wl.N, wl.K)
    th, b, upd = wl.theta.clone(), wl.momentum.clone(), torch.empty_like(wl.theta)
    assert plan.outer_step(th, b, wl.replicas, iso.make_opts(1.0, 0.7, 0.9, sync=True), update_out=upd) == 0
    ref = oracle_step(wl.table, wl.theta, wl.momentum, wl.replicas, 1.0, 0.7, 0.9)
    ref["theta_in"] = wl.theta.double().cpu().numpy()
    check_step(wl.table, th.double().cpu().numpy(), b.double().cpu().numpy(), upd.double().cpu().numpy(),
               plan.read_diag()["sigma_bar"], ref)
    th2, b2, upd2 = captured_step(plan, iso, wl)
    assert torch.equal(th, th2) and torch.equal(b, b2) and torch.equal(upd, upd2)
