"""Toeplitz sampling in the mixed forms: tiles read out of strips of core
matrices.

Sampling with unit vectors returns the entries, so S^r is A - D^(L) and S^c its
transpose, to the 24 (BF16 x 3, exact) or 22 bits (TF32 x 2) that the terms
hold.  Orders around a tile of 128 rows, a k-tile of 32 or 64 and a strip, one
column tile of 64 or 128 and several, leaves that straddle tiles, a matrix that
differs from its transpose, and K split over CTAs."""
import numpy as np
import pytest

import workloads as w
from oracle import tree as otree

import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hss():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1810_04125_gb300 import build, hss as h
    build.build()
    return h


@pytest.mark.parametrize("precision", ["bf16x3", "tf32x2"])
@pytest.mark.parametrize("n,leaf,cols", [(1, 1, 1), (33, 8, 33), (127, 40, 64), (129, 16, 129), (300, 70, 300),
                                         (1027, 128, 130), (9000, 256, 8),
                                         (9001, 256, 100)])
def test_entries(hss, precision, n, leaf, cols):
    import torch
    rng = np.random.default_rng(n)
    col, row = rng.standard_normal(n), rng.standard_normal(n)
    row[0] = col[0]
    at = rng.permutation(n)[:cols]      # column j of R is e_at[j]
    R = np.zeros((n, cols))
    R[at, np.arange(cols)] = 1.0
    S = [torch.full((n, cols), float("nan"), dtype=torch.float64, device=gu.dev()) for _ in range(2)]
    hss.hss_sample_offdiag(gu.device_source(w.Source(w.SRC_TOEPLITZ, n, col=col, row=row)), leaf, gu.PREC[precision],
                           gu.col_major(R), S[0], S[1])
    torch.cuda.synchronize()
    leaf_of = np.zeros(n, int)
    for q, t in enumerate(t for t in otree.halving_tree(n, leaf) if t.is_leaf):
        leaf_of[t.I] = q
    i, j = np.arange(n)[:, None], at[None, :]
    off = leaf_of[i] != leaf_of[j]
    d = i - j
    A = np.where(d >= 0, col[np.abs(d)], row[np.abs(d)])       # A(i, at[j])
    T = np.where(d <= 0, col[np.abs(d)], row[np.abs(d)])       # A(at[j], i)
    for s, E in ((S[0], A), (S[1], T)):
        E = np.where(off, E, 0.0)
        g = s.cpu().numpy()
        if precision == "bf16x3":
            assert np.array_equal(g, E.astype(np.float32).astype(np.float64))
        else:
            assert np.all(np.abs(g - E) <= 2.0 ** -21 * np.abs(E))
