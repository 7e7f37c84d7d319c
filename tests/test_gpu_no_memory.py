"""What needs no memory of its own does not fail for want of it: the digits of
the exact-split products are used where they can be allocated."""
import pytest

import fake_alloc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


WIDE_PRODUCT = r"""
n = 1500
P = w.uniform_points(n, 3, seed=2)
P = P[hss.hss_rcb_order(P, 100)]
A = w.gaussian_kernel(P, 1.0, 0.5).to_dense()
H = hss.hss_compress(gu.device_source(w.dense_source(A)), hss.make_opts(100, 1e-9, 1e-12, 64, 64, n, hss.HSS_DOUBLING))
X = gu.col_major(np.random.default_rng(1).standard_normal((n, 1600)))
for tr in (False, True):
    Y, Z = (torch.empty((1600, n), dtype=torch.float64, device=gu.dev()).t() for _ in range(2))
    hss.hss_matvec(H, X, Y, transpose=tr)
    before = fake.fake_refused()
    fake.fake_largest(1 << 20, 1)   # the node vectors' buffer, but no digits
    hss.hss_matvec(H, X, Z, transpose=tr)
    torch.cuda.synchronize()
    fake.fake_largest(-1, 0)
    assert fake.fake_refused() > before
    d = (Y - Z).abs().cpu().numpy()
    # the same sums of at most n terms in FP64, over the levels
    assert np.all(d <= 1e-12 * (np.abs(A).sum(axis=1).max() * np.abs(X.cpu().numpy()).max())), d.max()
"""


def test_wide_product_without_digits(tmp_path):
    fake_alloc.run(WIDE_PRODUCT, tmp_path)


MANY_COLUMNS = r"""
n, nc = 4096, 70000   # digits of R: 4.6 GB
src = gu.device_source(w.toeplitz_cos(n))
R = torch.randn((nc, n), dtype=torch.float64, device=gu.dev(), generator=torch.Generator(device=gu.dev()).manual_seed(1)).t()
S = [torch.full((n, nc), float("nan"), dtype=torch.float64, device=gu.dev()) for _ in range(2)]
T = [torch.empty((n, 100), dtype=torch.float64, device=gu.dev()) for _ in range(2)]
held = fake.fake_held()
fake.fake_peak(1)
hss.hss_sample_offdiag(src, 128, 0, R, *S)
torch.cuda.synchronize()
assert fake.fake_peak(1) - held < 5e9, fake.fake_peak(0)   # two caps of 2^31 bytes, and bookkeeping
for c in (0, 32700, 65400, nc - 100):   # slabs of 32768
    hss.hss_sample_offdiag(src, 128, 0, R[:, c:c + 100], *T)
    assert all(torch.equal(s[:, c:c + 100], t) for s, t in zip(S, T))
"""


def test_digits_of_many_columns(tmp_path):
    fake_alloc.run(MANY_COLUMNS, tmp_path)


COMPRESSION = r"""
import gc
n, leaf = 4096, 64
P = w.uniform_points(n, 3, seed=2)
P = gu.col_major(P[hss.hss_rcb_order(P, leaf)])
src = hss.points_source(w.SRC_GAUSS, P, 0.5, 1.0)
X = gu.col_major(np.random.default_rng(1).standard_normal((n, 3)))

def compress():
    hss.hss_release_cached()
    gc.collect()
    H = hss.hss_compress(src, hss.make_opts(leaf, 1e-6, 1e-10, 64, 64, 2048, hss.HSS_DOUBLING))
    Y = torch.empty((3, n), dtype=torch.float64, device=gu.dev()).t()
    hss.hss_matvec(H, X, Y)
    return H.ranks(), Y.cpu().numpy()

compress()
hss.hss_release_cached()
held = fake.fake_held()
fake.fake_peak(1)
ranks, Y = compress()
peak = fake.fake_peak(1) - held
digits = 16 * n * n
hss.hss_release_cached()
fake.fake_budget(peak - digits * 8 // 10 - (fake.fake_held() - held))
before = fake.fake_refused()
ranks2, Z = compress()
assert fake.fake_refused() > before
assert ranks == ranks2
assert np.linalg.norm(Y - Z) <= 1e-12 * np.linalg.norm(Y), np.linalg.norm(Y - Z) / np.linalg.norm(Y)
"""


def test_compression_gives_its_digits_back(tmp_path):
    """A compression that fits without the digits it keeps for speed fits."""
    fake_alloc.run(COMPRESSION, tmp_path)


ENTRIES = r"""
n = 6000   # one leaf: its block fills the handle's last chunk of memory
A = w.toeplitz_cos(n).to_dense()
src = gu.device_source(w.dense_source(A))
H = hss.hss_compress(src, hss.make_opts(n, 1e-6, 1e-10, 16, 16, 16, hss.HSS_DOUBLING))
I, J = (torch.arange(k, n, 997, device=gu.dev(), dtype=torch.int32) for k in (0, 5))
out = torch.empty((J.numel(), I.numel()), dtype=torch.float64, device=gu.dev()).t()
X = gu.col_major(np.eye(n)[:, :3])
Y = torch.empty((3, n), dtype=torch.float64, device=gu.dev()).t()
fake.fake_budget(64 << 20)
hss.hss_get_entries(H, I, J, out)
hss.hss_matvec(H, X, Y)
torch.cuda.synchronize()
assert np.array_equal(out.cpu().numpy(), A[np.ix_(I.cpu().numpy(), J.cpu().numpy())])
assert np.array_equal(Y.cpu().numpy(), A[:, :3])
held = fake.fake_held()
fake.fake_budget(0)
for call in (lambda: hss.hss_get_entries(H, I, J, out), lambda: hss.hss_matvec(H, X, Y)):
    try:
        call()
    except hss.HSSError as e:
        assert e.status in (2, 3)
assert fake.fake_held() == held
"""


def test_tables_of_a_handle(tmp_path):
    """The first entries of a handle take memory of their own size, not a chunk."""
    fake_alloc.run(ENTRIES, tmp_path)


TOEPLITZ = r"""
n = 4096   # one orientation of the packed terms: 134 MB, both: 268
src = hss.toeplitz_source(torch.from_numpy(w.toeplitz_cos(n).col).to(gu.dev()))
opts = hss.make_opts(128, 1e-4, 1e-8, 128, 128, 1024, hss.HSS_DOUBLING, hss.HSS_PREC_TF32X2)
hss.hss_compress(src, opts)
bytes_ = []
for free in (4 << 30, 500 << 20):   # 0.4 of it: room for both, for one
    hss.hss_release_cached()
    fake.fake_free(free)
    st = hss.hss_compress(src, opts).stats()
    fake.fake_free(-1)
    bytes_.append(st.bytes_sample - 16.0 * n * st.d_final)
print(bytes_)
assert bytes_[0] > 0 and bytes_[1] == 0   # A's own traffic, counted where it is packed
"""


def test_toeplitz_is_not_packed_where_one_orientation_fits(tmp_path):
    fake_alloc.run(TOEPLITZ, tmp_path)


LAPLACE = r"""
n, nc = 3000, 64
P = w.laplace_kernel(w.uniform_points(n, 3, seed=2)).points
src = hss.points_source(w.SRC_LAPLACE, gu.col_major(P[hss.hss_rcb_order(P, 100)]), 1.0)
R = gu.col_major(w.gaussian_matrix(1, n, 0, nc))
tiles = 3 * 16384 * -(-n // 128) * -(-n // 64)   # the packed matrix
out = []
for over in (None, tiles - 60000, 0, -60000):   # all; tiles at the cost of what comes after; no tiles; no split points either
    S = [torch.full((n, nc), float("nan"), dtype=torch.float64, device=gu.dev()) for _ in range(2)]
    if over is not None:   # leaf table, rounded R, packed R, split points
        fake.fake_budget(4 * n + 8 * n * nc + 4 + 128 * 64 * -(-n // 64) + 32 * n + 1000 + over)
    hss.hss_sample_offdiag(src, 100, hss.HSS_PREC_BF16X3, R, *S)
    torch.cuda.synchronize()
    fake.fake_budget(-1)
    out.append(S)
assert fake.fake_refused() >= 3
assert all(torch.equal(a, b) for S in out[1:] for a, b in zip(S, out[0]))
"""


def test_mixed_samples_without_packed_tiles(tmp_path):
    """Tiles and split points are for speed: the samples are the same bits."""
    fake_alloc.run(LAPLACE, tmp_path)
