"""The exact-split FP64 products (k_gemm_xs.cu) at the edges of their tiles,
k-tiles and chains, against products in extended precision.

Tolerance: one rounding of the result to FP64, plus what the digits leave out:
per term 2^-62 of (largest element of the row) x (largest of the column) from
either operand's tail and from the products below the last digit weight, taken
as 2^-60 for all of them together."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu

LD = np.longdouble


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1810_04125_gb300 import build
    build.build()
    return t


def _leaf_mask(n, leaf):
    lab, stack = np.zeros(n, int), [(0, n)]
    while stack:
        a, m = stack.pop()
        if m <= leaf:
            lab[a:a + m] = a
        else:
            stack += [(a, m // 2), (a + m // 2, m - m // 2)]
    return lab[:, None] == lab[None, :]


def _check(S, A, R):
    E = A.astype(LD) @ R.astype(LD)
    tail = A.shape[1] * 2.0 ** -60 * np.abs(A).max(axis=1)[:, None] * np.abs(R).max(axis=0)[None, :]
    bound = 2.0 ** -53 * np.abs(E) * (1 + 2.0 ** -20) + tail
    assert np.all(np.abs(S - E) <= bound), float((np.abs(S - E) / (bound + 1e-300)).max())


def _sample(torch, src, leaf, R):
    from paper_1810_04125_gb300 import hss
    import gpu_util as gu
    n, nc = R.shape
    out = [torch.full((n, nc), float("nan"), dtype=torch.float64, device=gu.dev()) for _ in range(2)]
    hss.hss_sample_offdiag(gu.device_source(src), leaf, 0, gu.col_major(R), *out)
    torch.cuda.synchronize()
    return [x.cpu().numpy() for x in out]


def _points(n, dim, leaf):
    from paper_1810_04125_gb300 import hss
    P = w.uniform_points(n, dim, seed=n)
    return P[hss.hss_rcb_order(P, leaf)]


# smallest order of the path, one past tile edges, tails of K of 1 and 31, an
# uneven tree (leaves on two levels), more column tiles than one, every source
@pytest.mark.parametrize("kind,n,leaf,nc", [
    ("dense", 192, 64, 1), ("dense", 193, 50, 64), ("dense", 255, 64, 65), ("dense", 257, 300, 3),
    ("dense", 384, 100, 130), ("dense", 513, 33, 63), ("toeplitz", 416, 64, 40), ("toeplitz_nonsym", 321, 40, 17),
    ("gauss", 300, 64, 33), ("laplace", 260, 64, 20), ("dense", 1027, 128, 5)])
def test_sampling(torch, kind, n, leaf, nc):
    rng = np.random.default_rng(n)
    src = {"dense": lambda: w.dense_source(rng.standard_normal((n, n)) * 10.0 ** rng.uniform(-20, 20, (n, 1))),
           "toeplitz": lambda: w.toeplitz_cos(n), "toeplitz_nonsym": lambda: w.toeplitz_nonsymmetric(n),
           "gauss": lambda: w.gaussian_kernel(_points(n, 3, leaf), 0.5, 1.0),
           "laplace": lambda: w.laplace_kernel(_points(n, 3, leaf))}[kind]()
    R = w.gaussian_matrix(7, n, 0, nc)
    Sr, Sc = _sample(torch, src, leaf, R)
    if kind in ("gauss", "laplace"):   # entries by the device's functions: FP64's own accuracy only
        A = src.to_dense()
        A[_leaf_mask(n, leaf)] = 0.0
        b = 1e-14 * (np.abs(A) @ np.abs(R)) + 1e-300
        assert np.all(np.abs(Sr - A @ R) <= b) and np.array_equal(Sr, Sc)
        return
    A = src.to_dense().copy()
    A[_leaf_mask(n, leaf)] = 0.0
    _check(Sr, A, R)
    _check(Sc, A.T, R)


def test_operands_the_digits_cannot_hold(torch):
    """A sparse R (columns of the identity) and non-finite entries take FP64
    FMAs: single entries come back as they are, NaN and Inf where IEEE puts
    them."""
    n, leaf = 300, 64
    rng = np.random.default_rng(1)
    A = rng.standard_normal((n, n)) * 10.0 ** rng.uniform(-30, 30, (n, n))
    A0 = np.where(_leaf_mask(n, leaf), 0.0, A)
    R = np.zeros((n, 40))
    R[7 * np.arange(40), np.arange(40)] = 1.0
    Sr, Sc = _sample(torch, w.dense_source(A), leaf, R)
    assert np.array_equal(Sr, A0[:, 7 * np.arange(40)]) and np.array_equal(Sc, A0[7 * np.arange(40)].T)
    A[3, 250], A[5, 200] = np.nan, np.inf
    R = np.abs(w.gaussian_matrix(2, n, 0, 10))
    Sr, Sc = _sample(torch, w.dense_source(A), leaf, R)
    assert np.isnan(Sr[3]).all() and np.isposinf(Sr[5]).all() and np.isfinite(np.delete(Sr, [3, 5], 0)).all()
    assert np.isnan(Sc[250]).all() and np.isposinf(Sc[200]).all() and np.isfinite(np.delete(Sc, [250, 200], 0)).all()


@pytest.mark.parametrize("nrhs,transpose", [(65, False), (200, True)])
def test_product_columns(torch, nrhs, transpose):
    """The wide HSS product: a column of X that the digits cannot hold (one
    entry; Inf) changes no other column, and every column is the single
    product's."""
    from paper_1810_04125_gb300 import hss
    import gpu_util as gu
    n = 900
    src = w.gaussian_kernel(_points(n, 3, 64), 1.0, 0.5)
    H = hss.hss_compress(gu.device_source(src), hss.make_opts(64, 1e-6, 1e-12, 64, 64, n, hss.HSS_DOUBLING))
    X = np.random.default_rng(3).standard_normal((n, nrhs))
    X[:, 10] = 0.0
    X[77, 10] = 1.0
    X[5, 20] = np.inf
    Xd = gu.col_major(X)
    Y = torch.empty((nrhs, n), dtype=torch.float64, device=gu.dev()).t()
    hss.hss_matvec(H, Xd, Y, transpose=transpose)
    one = torch.empty((1, n), dtype=torch.float64, device=gu.dev()).t()
    for j in (0, 9, 10, 20, 63, 64, nrhs - 1):
        hss.hss_matvec(H, Xd[:, j:j + 1], one, transpose=transpose)
        a, b = Y[:, j].cpu().numpy(), one[:, 0].cpu().numpy()
        if j == 20:
            assert np.array_equal(np.isfinite(a), np.isfinite(b)) and not np.isfinite(a).all()
        else:   # both within a few hundred roundings of terms bounded by |H||x|
            assert np.abs(a - b).max() <= 1e-13 * np.abs(src.to_dense()).sum(axis=1).max() * np.abs(X[:, j]).max()


# columns that the digits cannot hold, with the rows of a tile shared by 8, 4, 2
# and 1 CTAs (as the columns make more tiles): against the same product by tasks,
# both sums of the same terms in FP64
@pytest.mark.parametrize("nrhs", [256, 640, 1300, 2600])
def test_shared_rows(torch, nrhs):
    from paper_1810_04125_gb300 import hss
    import gpu_util as gu
    n = 800
    src = w.dense_source(np.random.default_rng(1).standard_normal((n, n)))
    H = hss.hss_compress(gu.device_source(src), hss.make_opts(100, 1e-12, 1e-13, 64, 64, n, hss.HSS_DOUBLING))
    rng = np.random.default_rng(5)
    X = gu.col_major(rng.standard_normal((n, nrhs)) * 10.0 ** -rng.uniform(0, 12, (n, 1)))
    Y, Z = (torch.empty((nrhs, n), dtype=torch.float64, device=gu.dev()).t() for _ in range(2))
    hss.hss_matvec(H, X, Y)
    for j in range(0, nrhs, 4):
        hss.hss_matvec(H, X[:, j:j + 4], Z[:, j:j + 4])
    bound = 1e-13 * np.abs(src.to_dense()).sum(axis=1).max() * np.abs(X.cpu().numpy()).max(axis=0)
    assert np.all(np.abs((Y - Z).cpu().numpy()) <= bound)
