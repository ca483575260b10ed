"""A tile's sums are added in the order of its columns, however the epilogue's two halves share
the stores of a partly filled tile: columns of zeros appended to a matrix (its last tile then
is a full one) only add zeros to every sum, and no bit of the result may change."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def iso():
    from paper_2607_03011_gb300 import isoloco
    isoloco.lib()
    return isoloco


def step(iso, mats, **kw):
    """U of each matrix (Delta as given) and the matrices' sigma_bar."""
    table, off = [], 0
    for m in mats:
        table.append((off, *m.shape))
        off += m.numel()
    rep = torch.cat([-m.reshape(-1) for m in mats])
    theta, mom, upd = (torch.zeros(off, device="cuda") for _ in range(3))
    plan = iso.Plan(table, off, 1)
    assert plan.outer_step(theta, mom, [rep], iso.make_opts(sync=True, **kw), update_out=upd) == 0
    return [upd[o:o + r * c].view(r, c) for o, r, c in table], plan.read_diag()["sigma_bar"]


def matrices(rows, cols, count, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return [torch.randn(rows, cols, generator=g, device="cuda") * 1e-3 for _ in range(count)]


def pad(m, cols):
    return torch.cat([m, m.new_zeros(m.shape[0], cols - m.shape[1])], 1)


@pytest.mark.parametrize("n", [64, 96, 128, 160, 192, 224])
def test_gram_sums(iso, n):
    """The normalisation comes from the Gram's sum of squares.  Fixed steps (no test whose result
    the appended zero directions could change) and the spectral scale, here 1 for the padded
    matrix, so that alpha makes both factors the same.  (Whole blocks of 32 columns: a block cut
    short adds its squares one by one.)"""
    mats = matrices(256, n, 24, n)
    scale = float(np.sqrt(np.float32(256) / np.float32(n)))
    want, _ = step(iso, [pad(m, 256) for m in mats], fast_steps=5, scale_kind=1, alpha=scale)
    got, _ = step(iso, mats, fast_steps=5, scale_kind=1)
    for w, g in zip(want, got):
        assert torch.equal(w[:, :n], g)


@pytest.mark.parametrize("cols", [70, 96, 100, 128, 129, 192, 250])
def test_trace(iso, cols):
    """sigma_bar comes from tr(Q^T Delta), summed by the tiles that write Q (here along the rows
    of wide matrices, whose Gram does not see the appended columns)."""
    mats = matrices(64, cols, 6, cols)
    want, want_sigma = step(iso, [pad(m, 256) for m in mats])
    got, got_sigma = step(iso, mats)
    assert got_sigma == want_sigma
    for w, g in zip(want, got):
        assert torch.equal(w[:, :cols], g)
