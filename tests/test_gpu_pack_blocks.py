"""Dense A in the mixed forms: the tiles packed by 128 x 128 blocks.

Sampling with unit vectors returns the entries: three BF16 terms hold an FP32
value exactly, so S^r is A - D^(L) rounded once to FP32 and S^c its transpose,
bit for bit (values below the normal FP32 range to 2^-126); two TF32 terms keep
22 bits.  Sizes at the edges of a block and of a k-tile, a leading dimension
larger than n, leaves that straddle blocks, and each side alone."""
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


def _values(n, rng):
    A = rng.standard_normal((n, n)) * 2.0 ** rng.integers(-90, 90, (n, n))
    k = A.size // 8
    at = rng.permutation(A.size)
    f = A.ravel()
    f[at[:k]] = 0.0
    f[at[k:2 * k]] *= 2.0 ** -60                                     # some below 2^-126
    x = f[at[2 * k:4 * k]].astype(np.float32)
    f[at[2 * k:4 * k]] = 0.5 * (x.astype(np.float64) + np.nextafter(x, np.float32(np.inf)))   # ties
    return A


@pytest.mark.parametrize("precision", ["bf16x3", "tf32x2"])
@pytest.mark.parametrize("n,leaf", [(1, 1), (31, 8), (127, 40), (128, 32), (129, 16), (321, 100), (700, 300)])
def test_entries(hss, precision, n, leaf):
    import torch
    A = _values(n, np.random.default_rng(n))
    src = gu.device_source(w.dense_source(A))
    R = gu.col_major(np.eye(n))
    S = [torch.full((n, n), float("nan"), dtype=torch.float64, device=gu.dev()) for _ in range(4)]
    hss.hss_sample_offdiag(src, leaf, gu.PREC[precision], R, S[0], S[1])
    hss.hss_sample_offdiag(src, leaf, gu.PREC[precision], R, S[2], None)
    hss.hss_sample_offdiag(src, leaf, gu.PREC[precision], R, None, S[3])
    torch.cuda.synchronize()
    E = A.copy()
    for t in otree.halving_tree(n, leaf):
        if t.is_leaf:
            E[np.ix_(t.I, t.I)] = 0.0
    f = E.astype(np.float32).astype(np.float64)
    for s, ref, exact in ((S[0], f, E), (S[1], f.T, E.T)):
        g = s.cpu().numpy()
        if precision == "bf16x3":
            assert np.all(np.abs(g - ref) <= np.where(np.abs(ref) >= 2.0 ** -100, 0.0, 2.0 ** -126))
        else:
            assert np.all(np.abs(g - exact) <= 2.0 ** -21 * np.abs(exact) + 2.0 ** -126)
    assert torch.equal(S[0], S[2]) and torch.equal(S[1], S[3])
