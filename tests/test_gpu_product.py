"""The HSS product task by task (k_prod.cu) and the entry extraction against the
dense expansion of the exported generators: every column count at which the
launch shape changes, both directions, ragged and uneven trees, nodes of rank
zero and of full rank, a leading dimension above n, sums longer than one staged
piece."""
import numpy as np
import pytest

import workloads as w
from oracle import apply

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


def _blockdiag(n):
    """Off-diagonal blocks zero but for one leaf's row of the matrix."""
    A = np.eye(n)
    A[:40, :40] += 1.0
    return w.dense_source(A)


CASES = {
    "toeplitz": (lambda: w.toeplitz_nonsymmetric(700), 64, 1e-8),          # transposed differs
    "uneven": (lambda: w.toeplitz_cos(1027), 128, 1e-8),                  # leaves on two levels
    "full_rank": (lambda: w.dense_source(np.random.default_rng(1).standard_normal((330, 330))), 40, 1e-12),
    "rank_zero": (lambda: _blockdiag(300), 50, 1e-8),
    "one_leaf": (lambda: w.toeplitz_cos(45), 64, 1e-8),
}


@pytest.mark.parametrize("name", CASES)
def test_products_and_entries(hss, name):
    import torch

    import gpu_util as gu
    mk, leaf, rtol = CASES[name]
    src = mk()
    n = src.n
    H = hss.hss_compress(gu.device_source(src), hss.make_opts(leaf, rtol, 1e-13, 32, 32, n, hss.HSS_DOUBLING))
    E = apply.to_dense(gu.expand_exported(H, n, leaf)) if n > leaf else src.to_dense()
    # both sides sum the same terms in FP64, at most n of them per level
    bound = 1e-13 * np.abs(E).sum(axis=1).max()
    rng = np.random.default_rng(2)
    for nrhs in (1, 2, 3, 4, 5, 8, 9, 33):
        X = rng.standard_normal((n, nrhs))
        big = torch.zeros((nrhs, n + 3), dtype=torch.float64, device=gu.dev()).t()   # ld n + 3
        big[:n] = gu.col_major(X)
        out = torch.full((nrhs, n + 5), 7.0, dtype=torch.float64, device=gu.dev()).t()
        for tr in (False, True):
            hss.hss_matvec(H, big[:n], out[:n], transpose=tr)
            Y = out.cpu().numpy()
            assert np.abs(Y[:n] - (E.T if tr else E) @ X).max() <= bound * np.abs(X).max() and (Y[n:] == 7.0).all()
    for nr, nc in ((1, 1), (9, 33), (70, 5)):
        I, J = rng.integers(0, n, nr), rng.integers(0, n, nc)
        o = torch.empty((nc, nr), dtype=torch.float64, device=gu.dev()).t()
        hss.hss_get_entries(H, torch.from_numpy(I.astype(np.int32)).to(gu.dev()),
                            torch.from_numpy(J.astype(np.int32)).to(gu.dev()), o)
        assert np.abs(o.cpu().numpy() - E[np.ix_(I, J)]).max() <= 1e-13 * np.abs(E).max() * max(1, leaf)
