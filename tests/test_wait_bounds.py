"""The waits of the pipelined kernels, read from their source (a wait that runs out cannot be
provoked in them without breaking the kernel): those after a failure share one limit, and a
thread that gives up a wait for a queue slot says so."""
import os
import re

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2607_03011_gb300", "csrc")


def source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


@pytest.mark.parametrize("name", ["gemm.cu", "polar_loop.cu"])
def test_copies_in_flight_share_one_limit(name):
    src = source(name)
    assert "drain_barriers(" in src
    assert not re.search(r"\(void\)\s*mbar_wait\(&full", src)


@pytest.mark.parametrize("name", ["gemm.cu", "polar_loop.cu"])
def test_queue_waits_have_one_limit_and_raise(name):
    src = source(name)
    waits = [m for m in re.finditer(r"mbar_wait\(&tq_(?:empty|full)\[q\],[^;{]*", src)]
    assert len(waits) >= 4
    limits = {}
    for m in waits:
        kind = "empty" if "tq_empty" in m[0] else "full"
        limits.setdefault(kind, set()).add((re.search(r"(\d \* )?kWaitTimeoutNs", m[0]) or [""])[0])
        # what follows within the statement raises the error (directly, or through `good`)
        after = src[m.end():m.end() + 400]
        assert "kErrTimeout" in after or "good = false" in after, m[0]
    assert all(len(v) == 1 for v in limits.values()), limits
