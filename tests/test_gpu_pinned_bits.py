"""The results' bits over widths at the edges of tiles and of the epilogue's blocks, for the paths
that round differently (single-plane steps, three passes, fixed steps, clipped spectrum, merge).

golden/outer_step_bits.txt holds a digest per case.  A change that is meant to keep the bits has
to leave them; one that is meant to round differently replaces the file (run this module with
`write`), and its error against the oracle is what the parity tests check.
"""
import hashlib
import os

import numpy as np
import pytest
import torch

from conftest import GOLDEN

pytestmark = pytest.mark.gpu

FILE = os.path.join(GOLDEN, "outer_step_bits.txt")
WIDTHS = [7, 31, 63, 64, 95, 96, 127, 128, 160, 191, 255, 257, 287, 300, 319]
PATHS = {"iso": {}, "full": dict(full_precision=1), "fast1": dict(fast_steps=1, scale_kind=1), "fast4": dict(fast_steps=4),
         "clip_high": dict(spectrum_kind=1), "merge": None}


def values(n, seed):
    """n fp32 values in (-1, 1), whole multiples of 2^-23 (SplitMix64's mix of the index)."""
    z = np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15) + np.uint64(seed)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    z ^= z >> np.uint64(31)
    return torch.from_numpy(((z >> np.uint64(40)).astype(np.int64) - (1 << 23)).astype(np.float32) / (1 << 23))


def digest(iso, path, n):
    """Three matrices (tall, wide, square) of least dimension n, two workers."""
    table, off = [], 0
    for r, c in ((n + 41, n), (n, n + 41), (n, n)):
        table.append((off, r, c))
        off += r * c
    theta = (values(off, 1) * 2.0 ** -5).cuda()
    mom = (values(off, 2) * 2.0 ** -12).cuda()
    reps = [theta - (values(off, 3 + k) * 2.0 ** -11).cuda() for k in range(2)]
    out = torch.zeros_like(theta)
    plan = iso.Plan(table, off, 2)
    kw = PATHS[path]
    if kw is None:
        plan.iso_c_merge(theta, reps, 0.75, out)
        torch.cuda.synchronize()
        assert plan.last_status() == 0
    else:
        assert plan.outer_step(theta, mom, reps, iso.make_opts(outer_lr=0.5, momentum=0.875, sync=True, **kw),
                               update_out=out) == 0
    h = hashlib.sha256()
    for t in (theta, mom, out):
        h.update(t.cpu().numpy().tobytes())
    return h.hexdigest()[:24]


def cases():
    return [(p, n) for p in PATHS for n in WIDTHS]


@pytest.mark.parametrize("path,n", cases())
def test_bits(path, n):
    from paper_2607_03011_gb300 import isoloco as iso
    with open(FILE) as f:
        want = dict(line.split() for line in f if line.strip() and not line.startswith("#"))
    assert digest(iso, path, n) == want[f"{path}_{n}"]


if __name__ == "__main__":
    import sys

    from paper_2607_03011_gb300 import isoloco as iso_
    if sys.argv[1:] == ["write"]:
        with open(FILE, "w") as f:
            f.write("# path_width: first 24 hex digits of SHA-256 over theta, B and U (see test_gpu_pinned_bits.py)\n")
            for p, n in cases():
                f.write(f"{p}_{n} {digest(iso_, p, n)}\n")
