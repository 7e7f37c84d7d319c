"""Exact-split FP64 products whose results are sums of terms that are all small
against the scales of their row and column: the large entry of a row meets a
zero (or next to one) of the other operand.  Every result keeps the accuracy
of a sum of FP64 FMAs, (K + 2) 2^-53 sum |a b| (its bound, Higham, Accuracy and
Stability, 3.1), whatever its neighbours."""
import numpy as np
import pytest

import workloads as w
from test_gpu_exact_split import _leaf_mask, _points, _sample, torch  # noqa: F401

pytestmark = pytest.mark.gpu

LD = np.longdouble


def _check(S, A, R):
    E = A.astype(LD) @ R.astype(LD)
    bound = (A.shape[1] + 2) * 2.0 ** -53 * (np.abs(A).astype(LD) @ np.abs(R).astype(LD))
    bad = np.abs(S - E) > bound
    assert not bad.any(), (int(bad.sum()), float((np.abs(S - E) / (bound + 1e-300)).max()))


# scale of the other entries; columns of R (of 70) without the large entry's
# term: single elements of a tile, and most of it; rounds of 128 along K: two,
# three with a ragged one, six
@pytest.mark.parametrize("n", [200, 300, 700])
@pytest.mark.parametrize("s,zeros,value", [(1e-6, 3, 0.0), (1e-10, 50, 0.0), (1e-14, 3, 1e-9), (1e-20, 50, 0.0),
                                           (1e-20, 3, 0.0)])
def test_dense_rows_with_one_large_entry(torch, n, s, zeros, value):
    rng = np.random.default_rng(n)
    leaf, q = 50, n - 7
    A = s * rng.standard_normal((n, n))
    A[:, q] = 1.0
    R = w.gaussian_matrix(3, n, 0, 70)
    R[q, 5:5 + zeros] = value
    Sr, Sc = _sample(torch, w.dense_source(A), leaf, R)
    A[_leaf_mask(n, leaf)] = 0.0
    _check(Sr, A, R)
    _check(Sc, A.T, R)


@pytest.mark.parametrize("kind", ["toeplitz", "toeplitz_nonsym"])
def test_generated_rows_with_few_large_entries(torch, kind):
    n, leaf = 513, 64
    rng = np.random.default_rng(2)
    c, r = (1e-15 * rng.standard_normal(n) for _ in range(2))
    c[100], c[0] = 1.0, 3.0
    r[0] = c[0]
    src = w.Source(w.SRC_TOEPLITZ, n, col=c, row=r if kind == "toeplitz_nonsym" else c.copy())
    R = w.gaussian_matrix(4, n, 0, 90)
    R[rng.random(R.shape) < 0.03] = 0.0
    Sr, Sc = _sample(torch, src, leaf, R)
    A = src.to_dense()
    A[_leaf_mask(n, leaf)] = 0.0
    _check(Sr, A, R)
    _check(Sc, A.T, R)


def test_narrow_gaussian_kernel(torch):
    """Each row's nearest points alone count.  Against the FMA kernel on the same
    entries: each within its bound of the exact sum (and of the subnormal
    range's spacing a term)."""
    import gpu_util as gu
    from paper_1810_04125_gb300 import hss
    n, leaf, nc = 513, 64, 90
    src = w.gaussian_kernel(_points(n, 3, leaf), 0.01, 1.0)
    R = w.gaussian_matrix(4, n, 0, nc)
    R[np.random.default_rng(2).random(R.shape) < 0.03] = 0.0
    S = _sample(torch, src, leaf, R)
    ref = [torch.empty((n, nc), dtype=torch.float64, device=gu.dev()) for _ in range(2)]
    hss.hss_sample_offdiag_noalloc(gu.device_source(src), leaf, 0, gu.col_major(R), *ref)
    A = src.to_dense()
    A[_leaf_mask(n, leaf)] = 0.0
    bound = 2 * (n + 2) * 2.0 ** -53 * (np.abs(A) @ np.abs(R)) * (1 + 1e-9) + 2 * n * 2.0 ** -1073 * np.abs(R).max()
    for s, f in zip(S, ref):
        assert np.all(np.abs(s - f.cpu().numpy()) <= bound)


def test_gaussian_entries_around_powers_of_two(torch):
    """Entries within a few ulps of 2^-k, on both sides of it: the scale of a row
    holds all of them (against the FMA kernel, as above)."""
    import gpu_util as gu
    from paper_1810_04125_gb300 import hss
    m, leaf, nc = 256, 64, 70
    k = 1 + np.arange(m) % 7
    x = np.sqrt(2.0 * k * np.log(2.0)) * (1.0 + (np.arange(m) - m // 2) * 2.0 ** -53)
    P = np.stack([np.concatenate([1e-9 * np.arange(m) * 2.0 ** -30, x]), np.zeros(2 * m)], axis=1)
    src = w.gaussian_kernel(P, 1.0, 1.0)
    R = w.gaussian_matrix(4, 2 * m, 0, nc)
    S = _sample(torch, src, leaf, R)
    ref = [torch.empty((2 * m, nc), dtype=torch.float64, device=gu.dev()) for _ in range(2)]
    hss.hss_sample_offdiag_noalloc(gu.device_source(src), leaf, 0, gu.col_major(R), *ref)
    A = src.to_dense()
    A[_leaf_mask(2 * m, leaf)] = 0.0
    bound = 2 * (2 * m + 2) * 2.0 ** -53 * (np.abs(A) @ np.abs(R)) * (1 + 1e-9)
    for s, f in zip(S, ref):
        assert np.all(np.abs(s - f.cpu().numpy()) <= bound)


@pytest.mark.parametrize("nrhs,transpose", [(1000, False), (1000, True)])
def test_wide_product(torch, nrhs, transpose):
    """Diagonal entries of 1e13 against zeros of X: the rows of H X there are
    what the other columns of H give (1e13 2^-61 = 4e-6 against entries of 1)."""
    import gpu_util as gu
    from paper_1810_04125_gb300 import hss
    n = 1500
    A = w.gaussian_kernel(_points(n, 3, 100), 1.0, 0.5).to_dense()
    big = np.arange(3, n, 31)
    A[big, big] = 1e13
    H = hss.hss_compress(gu.device_source(w.dense_source(A)),
                         hss.make_opts(100, 1e-9, 1e-12, 64, 64, n, hss.HSS_DOUBLING))
    rng = np.random.default_rng(5)
    X = rng.standard_normal((n, nrhs))
    X[big[:, None], rng.integers(0, nrhs, (big.size, 20))] = 0.0
    Y = torch.empty((nrhs, n), dtype=torch.float64, device=gu.dev()).t()
    Z = torch.empty((4, n), dtype=torch.float64, device=gu.dev()).t()
    Xd = gu.col_major(X)
    hss.hss_matvec(H, Xd, Y, transpose=transpose)
    zero = X == 0.0
    for j in range(0, nrhs, 4):   # (four columns: FP64 FMAs)
        hss.hss_matvec(H, Xd[:, j:j + 4], Z, transpose=transpose)
        d = np.abs((Y[:, j:j + 4] - Z).cpu().numpy())[zero[:, j:j + 4]]
        assert d.size == 0 or d.max() <= 1e-11   # sums of 1500 terms of order 1, 2^-53 each, over ten levels
