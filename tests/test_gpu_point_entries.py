"""The FP32-pair evaluation of 1 / (4 pi |x - y|) in the mixed forms' kernels.

Sampling with unit vectors returns the matrix entries themselves: three BF16
terms hold an FP32 value exactly, so S is the entry rounded once to FP32.  The
expected value is that rounding of the FP64 formula; the two may differ, by one
unit in the last place, only where the FP64 value (2^-50 of it, plus the
rounding of coordinates that nearly cancel, 2^-51 max|coordinate| / r) lies
within 2^-40 of itself and of a rounding boundary.  In TF32 x 2 the entry keeps
22 bits: 2^-21 relative."""
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


def _points(form, n, rng):
    x = rng.random((n, 3))
    if form == "shifted":          # coordinates far larger than the distances
        x = 1000.0 + x
    elif form == "small":
        x = x * 1e-7
    elif form == "tiny":           # r^2 below the range of the FP32 path
        x = x * 1e-12
    elif form == "huge":           # ... and above it
        x = x * 1e12
    elif form == "clusters":       # neighbours at 1e-9 of the coordinates
        x = x[rng.integers(0, 8, n)] + 1e-9 * rng.random((n, 3))
    elif form == "line":
        x = np.column_stack([np.arange(n) / 64.0, np.zeros(n), np.zeros(n)])
    return np.asfortranarray(x)


@pytest.mark.parametrize("precision", ["bf16x3", "tf32x2"])
@pytest.mark.parametrize("form,n", [("cube", 1000), ("shifted", 515), ("small", 257), ("tiny", 200), ("huge", 200),
                                    ("clusters", 600), ("line", 300), ("cube", 130)])
def test_entries(hss, precision, form, n):
    import torch
    leaf = 32
    P = _points(form, n, np.random.default_rng(n))
    R = np.eye(n)
    Sr = torch.full((n, n), float("nan"), dtype=torch.float64, device=gu.dev())
    Sc = torch.full((n, n), float("nan"), dtype=torch.float64, device=gu.dev())
    hss.hss_sample_offdiag(gu.device_source(w.laplace_kernel(P)), leaf, gu.PREC[precision], gu.col_major(R), Sr, Sc)
    torch.cuda.synchronize()
    r2 = sum((P[:, None, c] - P[None, :, c]) ** 2 for c in range(3))
    off = np.ones((n, n), bool)
    for t in otree.halving_tree(n, leaf):
        if t.is_leaf:
            off[np.ix_(t.I, t.I)] = False
    r = np.sqrt(np.where(off, r2, 1.0))
    E = np.where(off, 1.0 / (4.0 * np.pi * r), 0.0)
    f = E.astype(np.float32)
    ulp = np.spacing(f).astype(np.float64)
    edge = 0.5 * ulp - np.abs(E - f.astype(np.float64))      # to the rounding boundary
    near = edge <= E * (2.0 ** -40 + 2.0 ** -50 * np.abs(P).max() / r)
    for S in (Sr.cpu().numpy(), Sc.cpu().numpy()):
        if precision == "bf16x3":
            assert np.all((S == f) | (near & (np.abs(S - f) <= ulp)))
        else:
            assert np.all(np.abs(S - E) <= 2.0 ** -21 * E)
