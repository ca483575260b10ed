"""TIES where the magnitudes of a worker lie close together (normalised or sign-like updates):
the trim's bracket has to hold no more of them than its buffer does, or four more passes over
the replicas follow."""
import numpy as np
import pytest
import torch

from oracle import merging

pytestmark = pytest.mark.gpu


def replicas(N, K, dtype, spread, seed):
    """theta = 0, |Delta| distinct within `spread` of one magnitude (0: normal values)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    out = []
    for _ in range(K):
        x = torch.randn(N, generator=g, device="cuda")
        if spread:
            x = x.sign() * (1.0 + spread * torch.rand(N, generator=g, device="cuda"))
        out.append((x * 1e-3).to(dtype))
    return out


def step(iso, plan, reps, N, s):
    theta, mom = torch.zeros(N, device="cuda"), torch.zeros(N, device="cuda")
    assert plan.diloco_outer_step(theta, mom, reps, iso.make_opts(sync=True, aggregator=1, sparsity=s)) == 0
    return theta, mom


@pytest.mark.parametrize("K", [3, 9])
@pytest.mark.parametrize("s", [0.1, 0.5])
@pytest.mark.parametrize("spread", [1e-3, 1e-2, 1.0])
def test_close_magnitudes_are_exact(spread, s, K):
    from paper_2607_03011_gb300 import isoloco as iso
    N = 300_001
    reps = replicas(N, K, torch.float32, spread, 5)
    plan = iso.Plan([(0, N, 0)], N, K)
    theta, mom = step(iso, plan, reps, N, s)
    zero = np.zeros(N, np.float32)
    ref = merging.merged_outer_step(zero, zero, [r.cpu().numpy() for r in reps], "ties", sparsity=s, seed=0, eta=0.7, mu=0.9)
    from test_gpu_merging import ties_check
    ties_check(mom.double().cpu().numpy(), ref["ties_parts"], K)


@pytest.mark.parametrize("spread", [1e-3, 5e-3])
def test_close_magnitudes_take_one_pass(spread):
    """The fallback's four passes would show in the trim's time: at these sizes a pass over the
    replicas (the bracket's, or one of the fallback's) is most of it."""
    from paper_2607_03011_gb300 import isoloco as iso
    N, K = 48_000_000, 4
    plan = iso.Plan([(0, N, 0)], N, K)

    def trim_ms(spread):
        reps = replicas(N, K, torch.float32, spread, 6)
        step(iso, plan, reps, N, 0.5)
        best = 1e9
        for _ in range(5):
            plan.profile(True)
            step(iso, plan, reps, N, 0.5)
            best = min(best, plan.profile_read()["trim"][0])
        plan.profile(False)
        return best

    spread_out, close = trim_ms(0.0), trim_ms(spread)
    print(f"trim: {spread_out:.3f} ms with normal magnitudes, {close:.3f} ms within {spread:g}")
    assert close < 2.0 * spread_out
