"""The product of a handle whose row and column ranks differ chooses its kernel
by the direction it runs in: H X of A and H^T X of A^T are the same sums and
change kernels at the same number of columns."""
import numpy as np
import pytest

import workloads as w
from test_gpu_product import hss  # noqa: F401

pytestmark = pytest.mark.gpu


def _one_row_rank(n, leaf):
    """Blocks p_i q_ij^T: a leaf's rows have rank 1, its columns rank n / leaf - 1."""
    rng = np.random.default_rng(7)
    m = n // leaf
    p = rng.standard_normal((m, leaf))
    A = np.concatenate([p[i][:, None] * rng.standard_normal(n)[None, :] for i in range(m)])
    for i in range(m):
        A[i * leaf:(i + 1) * leaf, i * leaf:(i + 1) * leaf] = rng.standard_normal((leaf, leaf))
    return A


def test_kernel_by_direction(hss, capfd, monkeypatch):
    import torch

    import gpu_util as gu
    n, leaf = 1024, 64
    A = _one_row_rank(n, leaf)
    Hs = [hss.hss_compress(gu.device_source(w.dense_source(M)), hss.make_opts(leaf, 1e-10, 1e-12, 64, 64, n, hss.HSS_DOUBLING))
          for M in (A, np.ascontiguousarray(A.T))]
    assert Hs[0].ranks() == {i: (c, r) for i, (r, c) in Hs[1].ranks().items()}
    assert max(r for r, _ in Hs[0].ranks().values()) < max(c for _, c in Hs[0].ranks().values())
    X, Y = (torch.randn((8192, n), dtype=torch.float64, device=gu.dev()).t() for _ in range(2))
    monkeypatch.setenv("HSS_TRACE", "1")

    def first_general(H, tr):   # the general path traces its launches, the task lists have none
        lo, hi = 1, 8192
        while lo < hi:
            mid = (lo + hi) // 2
            capfd.readouterr()
            hss.hss_matvec(H, X[:, :mid], Y[:, :mid], transpose=tr)
            torch.cuda.synchronize()
            if "hss trace" in capfd.readouterr().err:
                hi = mid
            else:
                lo = mid + 1
        return lo

    got = [[first_general(H, tr) for tr in (False, True)] for H in Hs]
    assert 1 < min(map(min, got)) and max(map(max, got)) < 8192
    assert got[0] == got[1][::-1], got
