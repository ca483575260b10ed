"""TIES and DARE over the worker counts at which their passes change shape: the last of a group
of eight workers whose bracket pass runs together, the first of the next one, and batches of
four that end early, with both replica types and an odd number of parameters."""
import numpy as np
import pytest
import torch

from oracle import merging
from paper_2607_03011_gb300 import workloads as W
from test_gpu_merging import check, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def iso():
    from paper_2607_03011_gb300 import isoloco
    isoloco.lib()
    return isoloco


@pytest.mark.parametrize("agg", ["ties", "dare"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("K", [7, 8, 9, 17])
def test_worker_groups(iso, K, dtype, agg):
    spec = W.custom_spec([("m", 300, 257), ("v", 9, 0)], K=K, rank=2, replica_dtype=dtype)
    wl = W.make_workload(spec, seed=40 + K, device="cuda")
    th_in = wl.theta.cpu().numpy()
    rc, th, b = run(iso, wl, agg, 0.3)
    assert rc == 0
    ref = merging.merged_outer_step(th_in, np.zeros(wl.N, np.float32), W.replicas_as_numpy(wl.replicas), agg,
                                    sparsity=0.3, seed=1234, eta=0.7, mu=0.9)
    check(th, b, ref, th_in.astype(np.float64), agg, K=wl.K)
