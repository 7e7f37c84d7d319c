"""Performance cases: what users of this library have it do, through its public
Python entry points (paper_1810_04125_gb300.hss).

Kinds of case
  product   hss_matvec, H X or H^T X with a kept handle: the inner operation of
            an iterative solver (few right-hand sides) and the way H is
            expanded or checked (blocks of up to 2048)
  entries   hss_get_entries, H(I, J): element extraction from a kept handle, as
            a program does that compresses a matrix built from compressed ones
  sample    hss_sample_offdiag, (A - D) R and (A - D)^T R: the sampling step
            alone, in the precisions that callers choose
  compress  hss_compress and one product with the new handle (a compression
            is only of use through its products)
  batch     hss_compress_batched over matrices of uneven sizes, and one
            product with each handle

Products, compressions and batches are in the plain form, the default
precision, and the mixed forms are measured through their sampling: in a whole
compression in a mixed form, samples that agree only to the form's own 1e-7
leave pivots between equals, and a change in the last bit of any step gives
another compression, as good and different by the tolerance.

The matrices are the families of the workloads and tests: Toeplitz 1/(1+k) and
cos(w k)/(1+k) given by their coefficients, the Gaussian kernel in 3 and 8
dimensions (dense, or generated from the points), the Laplace single layer on a
sphere (generated), I + U D V^T with geometrically decaying D (dense).  The
seed changes the points or coefficients, the random matrix R and the operands.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1810_04125_gb300 import hss

PREC = {"fp64": hss.HSS_PREC_FP64, "tf32x2": hss.HSS_PREC_TF32X2, "bf16x3": hss.HSS_PREC_BF16X3}
STRAT = {"doubling": hss.HSS_DOUBLING, "incrementing": hss.HSS_INCREMENTING}
F64 = torch.float64
DEV = "cuda"


def _case(name, kind, matrix, n, leaf, rtol, atol, strategy, d0, dd, d_max, precision, **more):
    c = dict(kind=kind, matrix=matrix, n=n, leaf=leaf, rtol=rtol, atol=atol, strategy=strategy, d0=d0, dd=dd,
             d_max=d_max, precision=precision, symmetric=False)
    c.update(more)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # a solver's inner product on the smallest benchmark matrix: one vector, latency alone
        _case("product_toeplitz_n1024_1", "product", "toeplitz", 1024, 64, 1e-6, 1e-12, "incrementing", 64, 32, 1024,
              "fp64", nrhs=1, transpose=False),
        # a block Krylov step with H^T, ragged order and leaves, 48 vectors
        _case("product_t_gauss3_n5003_48", "product", "gauss3", 5003, 100, 1e-6, 1e-12, "doubling", 64, 64, 4096,
              "fp64", nrhs=48, transpose=True),
        # H applied to a wide block, as the expansion and the error check do; large ranks
        _case("product_gauss8_n4096_2048", "product", "gauss8_dense", 4096, 128, 1e-4, 1e-8, "doubling", 128, 128,
              4096, "fp64", nrhs=2048, transpose=False),
        # a block of entries of a compressed kernel matrix
        _case("entries_laplace_n3000", "entries", "laplace", 3000, 128, 1e-6, 1e-10, "incrementing", 64, 32, 3000,
              "fp64", nr=400, nc=300),
        # sampling alone, the plain form on a dense matrix of ragged order
        _case("sample_fp64_dense_n6001_200", "sample", "gauss8_dense", 6001, 128, 0.0, 0.0, "doubling", 200, 200, 200,
              "fp64"),
        # sampling alone, mixed form, entries generated from points
        _case("sample_bf16x3_laplace_n12000_128", "sample", "laplace", 12000, 256, 0.0, 0.0, "doubling", 128, 128, 128,
              "bf16x3"),
        # the first sampling pass of the benchmark workload: a dense matrix larger than L2, mixed form
        _case("sample_tf32x2_dense_n16384_128", "sample", "gauss8_dense", 16384, 128, 0.0, 0.0, "doubling", 128, 128,
              128, "tf32x2"),
        # the sampling of the largest configuration: entries from a coefficient table
        _case("sample_tf32x2_toeplitz_n131072", "sample", "toeplitz_cos", 131072, 256, 0.0, 0.0, "doubling", 256, 256,
              256, "tf32x2"),
        # the smallest benchmark configuration: a compression of a few milliseconds
        _case("compress_toeplitz_n1024", "compress", "toeplitz", 1024, 64, 1e-6, 1e-12, "incrementing", 64, 32, 1024,
              "fp64", nrhs=8),
        # the benchmark's matrix family in the plain form (the default precision): Doubling, large ranks
        _case("compress_gauss8_n8192", "compress", "gauss8_dense", 8192, 128, 1e-4, 1e-8, "doubling", 128, 128, 4096,
              "fp64", nrhs=8),
        # the surface kernel: generated entries, many adaptations, the Incrementing test at a tight tolerance
        _case("compress_laplace_n4001", "compress", "laplace", 4001, 128, 1e-6, 1e-8, "incrementing", 128, 64, 4001,
              "fp64", nrhs=8),
        # many matrices of uneven sizes in one call
        _case("batch16_n1024_4000", "batch", "mixed", 4000, 128, 1e-5, 1e-8, "doubling", 64, 64, 4096, "fp64",
              count=16, n_min=1024, nrhs=4),
    ]


def _between(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product", "product", "entries", "sample", "sample", "compress", "compress", "batch"])
    leaf = rng.choice([64, 100, 128, 256])
    strategy = rng.choice(["doubling", "incrementing"])
    if kind == "product":
        m = rng.choice(["toeplitz", "gauss3", "gauss8_dense", "laplace"])
        n = _between(rng, 700, 5500)
        return _case(None, kind, m, n, leaf, 1e-4 if m == "gauss8_dense" else rng.choice([1e-4, 1e-6]), 1e-10, strategy,
                     64, 64, n, "fp64", nrhs=_between(rng, 1, 2048), transpose=rng.random() < 0.4)
    if kind == "entries":
        n = _between(rng, 700, 5500)
        return _case(None, kind, rng.choice(["toeplitz", "gauss3", "laplace"]), n, leaf, 1e-6, 1e-10, "incrementing",
                     64, 32, n, "fp64", nr=_between(rng, 10, 800), nc=_between(rng, 10, 800))
    if kind == "sample":
        m = rng.choice(["gauss8_dense", "udv_dense", "gauss3", "laplace", "toeplitz_cos"])
        w = _between(rng, 16, 512)
        precision = rng.choice(["fp64", "tf32x2", "bf16x3"])
        n = _between(rng, 1000, 50000 if m == "toeplitz_cos" and precision != "fp64" else 12000)
        return _case(None, kind, m, n, leaf, 0.0, 0.0, "doubling", w, w, w, precision)
    if kind == "batch":
        return _case(None, kind, "mixed", _between(rng, 2500, 4500), leaf, 1e-5, 1e-8, strategy, 64, 64, 4096, "fp64",
                     count=rng.randint(4, 16), n_min=_between(rng, 700, 1500), nrhs=4)
    m = rng.choice(["toeplitz", "toeplitz_cos", "gauss3", "gauss8_dense", "laplace", "udv_dense"])
    n = _between(rng, 700, 4500 if m in ("gauss3", "laplace") else 8192)
    return _case(None, kind, m, n, leaf, rng.choice([1e-4, 1e-6]) if m != "gauss8_dense" else 1e-4, 1e-8, strategy,
                 rng.choice([64, 96, 128]), rng.choice([32, 64]), min(n, 4096), "fp64",
                 symmetric=m != "udv_dense" and rng.random() < 0.3, nrhs=8)


# ------------------------------------------------------------------- inputs
def _points(matrix, n, leaf, seed):
    """The point set in the library's cluster order, n x dim on the device."""
    g = np.random.default_rng(seed)
    if matrix == "laplace":   # Fibonacci lattice of the unit sphere, rotated by the seed
        i = np.arange(n, dtype=np.float64)
        z = 1.0 - (2.0 * i + 1.0) / n
        r = np.sqrt(np.maximum(0.0, 1.0 - z * z))
        phi = i * (math.pi * (3.0 - math.sqrt(5.0)))
        q, _ = np.linalg.qr(g.standard_normal((3, 3)))
        P = np.stack([r * np.cos(phi), r * np.sin(phi), z], axis=1) @ q
    else:
        P = g.random((n, 8 if matrix.startswith("gauss8") else 3))
    P = P[hss.hss_rcb_order(P, leaf)]
    return torch.from_numpy(np.ascontiguousarray(P)).to(DEV)


def _laplace_diag(n):
    """Twice the term of the lattice's nearest distance, about 3.09 / sqrt(n)."""
    return 2.0 / (4.0 * math.pi * 3.09 / math.sqrt(n))


def _kernel_block(matrix, X, lo, hi):
    """Columns lo..hi of a kernel matrix, n x (hi - lo)."""
    n = X.shape[0]
    r2 = torch.zeros((n, hi - lo), dtype=F64, device=X.device)
    for c in range(X.shape[1]):
        r2 += (X[:, c:c + 1] - X[lo:hi, c][None, :]) ** 2
    d = torch.arange(lo, hi, device=X.device)
    if matrix == "laplace":
        r2[d, d - lo] = 1.0
        B = 1.0 / (4.0 * math.pi * torch.sqrt(r2))
        B[d, d - lo] = _laplace_diag(n)
    else:
        B = torch.exp(-r2 / 2.0)
        if matrix.startswith("gauss8"):
            B[d, d - lo] += 1.0   # the benchmark's shift
    return B


def _toeplitz(matrix, n, seed):
    k = torch.arange(n, dtype=F64, device=DEV)
    t = float(np.random.default_rng(seed).uniform(-0.01, 0.01))
    if matrix == "toeplitz":
        return (1.0 + t) / (1.0 + k)
    if matrix == "toeplitz_power":
        return (1.0 + k) ** (-(1.5 + t))
    return torch.cos((0.3 + t) * k) / (1.0 + k)


def _dense(matrix, n, leaf, seed):
    """A stored row-major as A^T (so that its transpose is column-major)."""
    At = torch.empty((n, n), dtype=F64, device=DEV)
    if matrix.startswith("udv"):
        g = torch.Generator(device=DEV).manual_seed(seed)
        r = max(8, n // 100)
        U, V = (torch.linalg.qr(torch.randn((n, r), dtype=F64, device=DEV, generator=g))[0] for _ in range(2))
        D = 2.0 ** (-53.0 * torch.arange(r, dtype=F64, device=DEV) / r)
        torch.mm(V * D, U.t(), out=At)
        At.diagonal().add_(1.0)
    elif matrix.startswith("toeplitz"):
        c = _toeplitz(matrix, n, seed)
        i = torch.arange(n, device=DEV)
        for lo in range(0, n, 1024):
            At[lo:lo + 1024] = c[(i[lo:lo + 1024, None] - i[None, :]).abs()]
    else:
        X = _points(matrix, n, leaf, seed)
        for lo in range(0, n, 1024):
            hi = min(n, lo + 1024)
            At[lo:hi] = _kernel_block(matrix, X, lo, hi).t()
    return At.t()


def _matrix(matrix, n, leaf, seed):
    """The data a program holds of A: a dense matrix, points or coefficients."""
    if matrix.endswith("_dense"):
        return _dense(matrix, n, leaf, seed)
    if matrix.startswith("toeplitz"):
        return _toeplitz(matrix, n, seed)
    return _points(matrix, n, leaf, seed).t().contiguous().t()   # column-major


def _source(matrix, data):
    if matrix.endswith("_dense"):
        return hss.dense_source(data)
    if matrix.startswith("toeplitz"):
        return hss.toeplitz_source(data)
    if matrix == "laplace":
        return hss.points_source(hss.HSS_SRC_LAPLACE, data, _laplace_diag(data.shape[0]))
    return hss.points_source(hss.HSS_SRC_GAUSS, data, 1.0, 0.0)


def _opts(c, seed):
    return hss.make_opts(c["leaf"], c["rtol"], c["atol"], c["d0"], c["dd"], min(c["d_max"], c["n"]),
                         STRAT[c["strategy"]], PREC[c["precision"]], 10, seed, symmetric=int(c["symmetric"]))


def _columns(n, w, seed):
    """n x w standard normal values, column-major."""
    g = torch.Generator(device=DEV).manual_seed(seed + 7)
    return torch.randn((w, n), dtype=F64, device=DEV, generator=g).t()


def _batch_members(c, seed):
    """(matrix, n) of every member: sizes log-uniform, Toeplitz and Gaussian kernels in turn."""
    g = np.random.default_rng(12345 + c["count"])   # the sizes belong to the case, not to the seed
    n = np.rint(np.exp(g.uniform(math.log(c["n_min"]), math.log(c["n"]), size=c["count"]))).astype(int)
    n[0] = c["n"]
    return [("toeplitz_power_dense" if i % 2 else "gauss3_dense", int(v)) for i, v in enumerate(n)]


def prepare(case, seed):
    c = case
    s = {"case": c}
    if c["kind"] == "batch":
        members = _batch_members(c, seed)
        s["data"] = [_dense(m[:-len("_dense")], n, c["leaf"], seed + 100 * i) for i, (m, n) in enumerate(members)]
        s["sources"] = [hss.dense_source(A) for A in s["data"]]
        s["opts"] = [_opts(dict(c, n=n), seed + i) for i, (_, n) in enumerate(members)]
        s["X"] = [_columns(n, c["nrhs"], seed + i) for i, (_, n) in enumerate(members)]
        return s
    n = c["n"]
    s["data"] = _matrix(c["matrix"], n, c["leaf"], seed)
    s["source"] = _source(c["matrix"], s["data"])
    if c["kind"] == "sample":
        w = c["d0"]
        s["R"] = _columns(n, w, seed)
        s["Sr"], s["Sc"] = (torch.empty((n, w), dtype=F64, device=DEV) for _ in range(2))
        return s
    s["opts"] = _opts(c, seed)
    if c["kind"] == "compress":
        s["X"] = _columns(n, c["nrhs"], seed)
        return s
    s["H"] = hss.hss_compress(s["source"], s["opts"])
    if c["kind"] == "product":
        s["X"] = _columns(n, c["nrhs"], seed)
        s["Y"] = torch.empty((c["nrhs"], n), dtype=F64, device=DEV).t()
    else:
        g = torch.Generator(device=DEV).manual_seed(seed)
        s["I"] = torch.randint(0, n, (c["nr"],), device=DEV, generator=g).to(torch.int32)
        s["J"] = torch.randint(0, n, (c["nc"],), device=DEV, generator=g).to(torch.int32)
        s["out"] = torch.empty((c["nc"], c["nr"]), dtype=F64, device=DEV).t()
    return s


def _apply(H, X):
    Y = torch.empty((X.shape[1], X.shape[0]), dtype=F64, device=DEV).t()
    hss.hss_matvec(H, X, Y)
    return Y


def run(state):
    s = state
    c = s["case"]
    if c["kind"] == "product":
        hss.hss_matvec(s["H"], s["X"], s["Y"], transpose=c["transpose"])
        return s["Y"]
    if c["kind"] == "entries":
        hss.hss_get_entries(s["H"], s["I"], s["J"], s["out"])
        return s["out"]
    if c["kind"] == "sample":
        hss.hss_sample_offdiag(s["source"], c["leaf"], PREC[c["precision"]], s["R"], s["Sr"], s["Sc"])
        return [s["Sr"], s["Sc"]]
    if c["kind"] == "compress":
        return _apply(hss.hss_compress(s["source"], s["opts"]), s["X"])
    return [_apply(H, X) for H, X in zip(hss.hss_compress_batched(s["sources"], s["opts"]), s["X"])]


def _data_bytes(matrix, n):
    if matrix.endswith("_dense"):
        return 8.0 * n * n
    return 8.0 * n * (1 if matrix.startswith("toeplitz") else 8 if matrix.startswith("gauss8") else 3)


def work(case):
    """Lower bounds that hold for any ranks: the diagonal blocks of a product,
    the first d0 columns of a compression's samples."""
    c = case
    n = float(c["n"])
    if c["kind"] == "product":
        return {"bytes": 8.0 * n * c["leaf"] / 2 + 16.0 * n * c["nrhs"], "flops": 2.0 * n * c["leaf"] / 2 * c["nrhs"]}
    if c["kind"] == "entries":
        return {"bytes": 4.0 * (c["nr"] + c["nc"]) + 8.0 * c["nr"] * c["nc"], "flops": 2.0 * c["nr"] * c["nc"]}
    if c["kind"] == "sample":
        return {"bytes": _data_bytes(c["matrix"], n) + 24.0 * n * c["d0"], "flops": 4.0 * n * n * c["d0"]}
    if c["kind"] == "compress":
        return {"bytes": _data_bytes(c["matrix"], n) + 16.0 * n * c["nrhs"],
                "flops": (2.0 if c["symmetric"] else 4.0) * n * n * c["d0"]}
    ns = [float(m) for _, m in _batch_members(c, 0)]
    return {"bytes": sum(8.0 * m * m + 16.0 * m * c["nrhs"] for m in ns), "flops": sum(4.0 * m * m * c["d0"] for m in ns)}


# -------------------------------------------------------------------- exact
def _leaf_of(n, leaf):
    """The leaf's first index for every index: a node of m > leaf splits into m // 2 and the rest."""
    lo = torch.zeros(n, dtype=torch.int64)
    stack = [(0, n)]
    while stack:
        a, m = stack.pop()
        if m <= leaf:
            lo[a:a + m] = a
        else:
            stack += [(a, m // 2), (a + m // 2, m - m // 2)]
    return lo.to(DEV)


def _block(matrix, data, lo, hi):
    """A(:, lo:hi)."""
    if matrix.endswith("_dense"):
        return data[:, lo:hi]
    if matrix.startswith("toeplitz"):
        i = torch.arange(data.shape[0], device=DEV)
        return data[(i[:, None] - i[None, lo:hi]).abs()]
    return _kernel_block("laplace" if matrix == "laplace" else "gauss", data, lo, hi)


def _times(matrix, data, X, transpose=False, leaf=0):
    """A X or A^T X, with the leaf diagonal blocks left out where leaf is given."""
    n = X.shape[0]
    label = _leaf_of(n, leaf) if leaf else None
    Y = torch.zeros((n, X.shape[1]), dtype=F64, device=DEV)
    for lo in range(0, n, 2048):
        hi = min(n, lo + 2048)
        B = _block(matrix, data, lo, hi)
        if leaf:
            B = torch.where(label[:, None] == label[None, lo:hi], 0.0, B)
        if transpose:
            Y[lo:hi] = B.t() @ X
        else:
            Y += B @ X[lo:hi]
    return Y


def _rounded(R, precision):
    """R as the mixed forms define it: rounded once to the significand of their operand type."""
    if precision == "fp64":
        return R
    s = 2048.0 if precision == "tf32x2" else 256.0
    m, e = torch.frexp(R)
    return torch.ldexp(torch.round(m * s) / s, e)


def exact(case, seed):
    c = case
    if c["kind"] == "batch":
        s = prepare(c, seed)
        return [_times("x_dense", A, X) for A, X in zip(s["data"], s["X"])]
    n = c["n"]
    data = _matrix(c["matrix"], n, c["leaf"], seed)
    if c["kind"] == "sample":
        R = _rounded(_columns(n, c["d0"], seed), c["precision"])
        return [_times(c["matrix"], data, R, t, c["leaf"]) for t in (False, True)]
    if c["kind"] == "entries":
        g = torch.Generator(device=DEV).manual_seed(seed)
        I = torch.randint(0, n, (c["nr"],), device=DEV, generator=g)
        J = torch.randint(0, n, (c["nc"],), device=DEV, generator=g)
        return _times(c["matrix"], data, torch.eye(n, dtype=F64, device=DEV)[:, J])[I]
    X = _columns(n, c["nrhs"], seed)
    if n > 40000:   # a symmetric Toeplitz matrix through its circulant of order 2 n
        z = torch.zeros(2 * n, dtype=F64, device=DEV)
        z[:n], z[n + 1:] = data, data[1:].flip(0)
        Z = torch.zeros((2 * n, X.shape[1]), dtype=F64, device=DEV)
        Z[:n] = X
        return torch.fft.irfft(torch.fft.rfft(z)[:, None] * torch.fft.rfft(Z, dim=0), n=2 * n, dim=0)[:n]
    return _times(c["matrix"], data, X, bool(c.get("transpose", False)))
