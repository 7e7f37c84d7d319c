"""A device wait of the exact-split product that runs out costs time, not the
result: calls that return before their work is done (hss_matvec, the FP64 form
of hss_sample_offdiag) give what they always give, and a compression, which
waits for its work, fails with HSS_ERR_TIMEOUT.

No wait is made to run out on the GPU: the library is built once more with
HSS_TEST_LOST_WAIT, where every other tile's last segment reports one after all
of its products are in."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import sys
sys.path[:0] = [{root!r}, {root!r} + "/tests"]
import numpy as np, torch
from paper_1810_04125_gb300 import build, hss
import gpu_util as gu, workloads as w

build.build()
ref = hss.lib()
build.OUT, build.LIB = {out!r}, {out!r} + "/libhss.so"
build.build(extra=["-DHSS_TEST_LOST_WAIT"])

def lost():
    hss._lib, hss.LIB_PATH = None, build.LIB
    return hss.lib()

test = lost()
n, leaf = 1500, 100
P = w.uniform_points(n, 3, seed=2)
hss._lib = ref
P = P[hss.hss_rcb_order(P, leaf)]
A = w.gaussian_kernel(P, 1.0, 0.5).to_dense()
A[np.arange(3, n, 31), np.arange(3, n, 31)] = 1e13   # (marked elements among the others)
src = gu.device_source(w.dense_source(A))
H = hss.hss_compress(src, hss.make_opts(leaf, 1e-9, 1e-12, 64, 64, n, hss.HSS_DOUBLING))
hss.hss_save(H, {out!r} + "/h.hss")
del H
X = np.random.default_rng(1).standard_normal((n, 1600))
X[3:n:31, 7:20] = 0.0
X[:, 600] *= 10.0 ** -np.random.default_rng(2).uniform(0, 12, n)
X = gu.col_major(X)
R = w.gaussian_matrix(5, n, 0, 150)
R[700, 3:5] = 0.0
R = gu.col_major(R)
got = []
for L in (ref, test):
    hss._lib = L
    G = hss.hss_load({out!r} + "/h.hss")
    out = []
    for tr in (False, True):
        Y = torch.empty((1600, n), dtype=torch.float64, device=gu.dev()).t()
        hss.hss_matvec(G, X, Y, transpose=tr)
        out.append(Y.cpu().numpy())
    S = [torch.full((n, 150), float("nan"), dtype=torch.float64, device=gu.dev()) for _ in range(2)]
    hss.hss_sample_offdiag(src, leaf, 0, R, *S)
    out += [s.cpu().numpy() for s in S]
    got.append(out)
    del G
scale = np.abs(A).sum(axis=1).max()
for k, (a, b) in enumerate(zip(*got)):
    assert np.isfinite(b).all()
    # sums of at most n terms in FP64, a few levels of them
    bound = 1e-12 * (np.abs(A) @ np.abs((X if k < 2 else R).cpu().numpy())) + 1e-12 * 6.0 * n
    assert np.all(np.abs(a - b) <= bound), (k, float((np.abs(a - b) / bound).max()))
    assert (a != b).any()   # (the tiles that were computed again)
hss._lib = test
try:
    hss.hss_compress(src, hss.make_opts(leaf, 1e-9, 1e-12, 64, 64, n, hss.HSS_DOUBLING))
    print("no error")
except hss.HSSError as e:
    print("status", e.status)
"""


def test_lost_wait(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    p = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT, out=str(tmp_path))], capture_output=True,
                       text=True, timeout=600)
    assert p.returncode == 0, p.stdout + p.stderr
    assert "status 6" in p.stdout, p.stdout
