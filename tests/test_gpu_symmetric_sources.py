"""Plain-form compressions of symmetric matrices take the row side alone
(sample_launches counts one product per pass instead of two): the same
result as the symmetric option, and no matrix that differs from its transpose
in a single bit is taken for symmetric."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hss():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1810_04125_gb300 import build
    build.build()
    from paper_1810_04125_gb300 import hss as h
    return h


def _run(hss, src, strategy, symmetric=0, precision=0):
    import torch

    import gpu_util as gu
    n = src.n
    o = hss.make_opts(50, 1e-6, 1e-12, 32, 16, n, strategy, precision, symmetric=symmetric)
    H = hss.hss_compress(gu.device_source(src), o)
    st = H.stats()
    X = gu.col_major(np.random.default_rng(0).standard_normal((n, 5)))
    out = []
    for tr in (False, True):
        Y = torch.empty((5, n), dtype=torch.float64, device=gu.dev()).t()
        hss.hss_matvec(H, X, Y, transpose=tr)
        out.append(Y.cpu().numpy())
    return out, st.sample_launches // (st.n_adapt + 1), st.flop_sample


def _points(hss, n):
    P = w.uniform_points(n, 3, seed=1)
    return P[hss.hss_rcb_order(P, 50)]


@pytest.mark.parametrize("kind", ["dense", "toeplitz", "gauss", "laplace"])
@pytest.mark.parametrize("strategy", [0, 1])
def test_symmetric_sources(hss, kind, strategy):
    n = 333
    src = {"dense": lambda: w.dense_source(w.gaussian_kernel(_points(hss, n), 0.3, 0.5).to_dense()),
           "toeplitz": lambda: w.Source(w.SRC_TOEPLITZ, n, col=1 / (1.0 + np.arange(n)), row=None),
           "gauss": lambda: w.gaussian_kernel(_points(hss, n), 0.3, 0.5),
           "laplace": lambda: w.laplace_kernel(_points(hss, n))}[kind]()
    if kind == "toeplitz":   # one table for both halves
        import torch

        import gpu_util as gu
        c = torch.from_numpy(src.col).to(gu.dev())
        src.row = src.col
        gu_source = gu.device_source
        try:
            gu.device_source = lambda s: hss.toeplitz_source(c)
            got, per, fl = _run(hss, src, strategy)
            ref, per2, fl2 = _run(hss, src, strategy, symmetric=1)
        finally:
            gu.device_source = gu_source
    else:
        got, per, fl = _run(hss, src, strategy)
        ref, per2, fl2 = _run(hss, src, strategy, symmetric=1)
    assert per == per2 == 1 and fl == 2 * fl2
    assert all(np.array_equal(a, b) for a, b in zip(got, ref))


# tile corners of the comparison (64 x 64) and both triangles
@pytest.mark.parametrize("i,j", [(0, 332), (63, 64), (64, 63), (332, 320), (127, 128), (1, 0)])
def test_one_bit_of_difference(hss, i, j):
    A = w.gaussian_kernel(_points(hss, 333), 0.3, 0.5).to_dense()
    A[i, j] = np.nextafter(A[i, j], 2.0)
    got, per, _ = _run(hss, w.dense_source(A), 0)
    assert per == 2
    X = np.random.default_rng(0).standard_normal((333, 5))
    for Y, B in zip(got, (A, A.T)):
        assert np.linalg.norm(Y - B @ X) <= 1e-5 * np.linalg.norm(B @ X)


def test_difference_in_every_tile(hss):
    """Tiles that see the flag set by others while they begin."""
    A = w.gaussian_kernel(_points(hss, 1900), 0.3, 0.5).to_dense()
    A += np.triu(1e-9 * np.random.default_rng(3).random(A.shape))
    got, per, _ = _run(hss, w.dense_source(A), 0)
    assert per == 2
    X = np.random.default_rng(0).standard_normal((1900, 5))
    for Y, B in zip(got, (A, A.T)):
        assert np.linalg.norm(Y - B @ X) <= 1e-5 * np.linalg.norm(B @ X)
