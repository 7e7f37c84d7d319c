// Entries of a compressed HSS matrix, H(I, J) for index sets I and J
// (section 2.1, eq. nestedUV): for i and j in one leaf, D(i, j); otherwise,
// with a and b the children of their lowest common ancestor tau that hold
// i and j,
//     H(i, j) = u_a(i) B_ab v_b(j)^T,
// where B_ab is tau's B12 (a first) or B21, and u_a(i) is row i of the
// nested basis of a: at a leaf the row of U = Pi [I; X^T] (eq. ID), one level
// up u_parent(i) = u_a(i) U_parent(rows of a's block, :) (the basis of a
// node is its children's bases times its own small one).  The same for
// v_b(j) with V.  A node that was not COMPRESSED (a partial result) keeps
// its blocks A(I_nu1, I_nu2), A(I_nu2, I_nu1) dense.
//
// Kept with the handle: the nodes, the inverse pivot orders of every node side
// and the leaf of every index.  A call is two kernels: one CTA per requested
// index walking its leaf's path to the root (row indices store W_i(level) =
// u_a(i) B_ab for every ancestor a, column indices v_b(j)), and a warp per
// eight entries finding the common ancestors and forming the dot products.
#include "hss_internal.h"

namespace hss {
namespace {

// inv[piv[q]] = q for every node side (one CTA per side)
__global__ void k_inv_piv(const EntryNode* __restrict__ nodes, int nn, int* __restrict__ err) {
  const int side = blockIdx.x & 1, id = blockIdx.x >> 1;
  if (id >= nn) return;
  const EntryNode& t = nodes[id];
  const int m = side ? t.mc : t.mr;
  const int* piv = side ? t.pivc : t.pivr;
  int* inv = side ? t.ipivc : t.ipivr;
  if (!piv || !inv) return;
  for (int q = threadIdx.x; q < m; q += blockDim.x) {
    const int p = piv[q];
    if (p < 0 || p >= m) { atomicCAS(err, 0, 2); continue; }
    inv[p] = q;
  }
}

// leaf_of[i] = the leaf that holds i (one CTA per node)
__global__ void k_leaf_of(const EntryNode* __restrict__ nodes, int* __restrict__ leaf_of) {
  const EntryNode& t = nodes[blockIdx.x];
  if (t.ch0 >= 0) return;
  for (int i = threadIdx.x; i < t.size; i += blockDim.x) leaf_of[t.lo + i] = blockIdx.x;
}

// Eight sums over a warp at once: lane l's a[x] are its parts of sum x; the
// return value is sum l / 4 (in all four lanes of that number).  Halving the
// number of sums with every exchange takes 9 additions where eight butterflies
// take 40 (an FP64 instruction of a warp occupies its scheduler's FP64 pipe
// for 64 clocks).
__device__ __forceinline__ double warp_sum8(double* a, int lane) {
#pragma unroll
  for (int h = 4; h >= 1; h /= 2) {
    const bool up = (lane & (4 * h)) != 0;
#pragma unroll
    for (int x = 0; x < h; ++x) {
      const double keep = up ? a[x + h] : a[x], give = up ? a[x] : a[x + h];
      a[x] = keep + __shfl_xor_sync(0xffffffffu, give, 4 * h);
    }
  }
  double s = a[0];
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  return s;
}

// Warps of a path CTA by the largest rank.  Walking a path is a chain of small
// products; with ranks of 100 and more four warps take several rounds of loads
// per block, and sixteen hide more of them (ranks to 200, Laplace n = 3000: one
// entry 448 us with 4 warps, 395 with 8, 219 with 16; 400 x 300 entries 854,
// 874, 731); with small ranks twelve of the sixteen only wait (Toeplitz n = 8192:
// 400 x 300 entries 104 us with 4 warps, 135 with 16).
inline int path_warps(int kcap) { return kcap >= 96 ? 16 : 4; }
constexpr int EW_MAX = 16;

// Row (CTAs below nr) or column vectors of the nested basis along the path of
// an index to the root.  A row stores W(level(a)) = u_a(i) B_ab for every
// ancestor a whose parent is COMPRESSED, a column v_a(j).  Wrow, Vcol:
// (count x (levels + 1) x kcap) doubles; shared memory 2 kcap doubles and, where
// they fit too (HAVE_SP), kcap ints for the positions, which are read from the
// tables again otherwise (ranks above 11600).  Bound by the FP64 pipe (sum of k_a k_b + k_a k_p per level) once the
// sums run along the blocks' contiguous direction: u B with eight columns of B
// per warp and lanes along u, u U_p with a lane per column.  Rows and columns
// go in one launch.
template <bool HAVE_SP>
__global__ void __launch_bounds__(32 * EW_MAX) k_entry_paths(const EntryNode* __restrict__ nodes,
                                                         const int* __restrict__ leaf_of, int n,
                                                         const int* __restrict__ I, int nr, const int* __restrict__ J,
                                                         double* __restrict__ Wrow, double* __restrict__ Vcol, int kcap,
                                                         int lp1, int* __restrict__ err) {
  extern __shared__ double sm[];
  double* u = sm;
  double* u2 = sm + kcap;
  int* sp = (int*)(sm + 2 * kcap);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32, EW = blockDim.x / 32;
  const int side = (int)blockIdx.x >= nr, r = side ? blockIdx.x - nr : blockIdx.x;
  const int i = side ? J[r] : I[r];
  if (i < 0 || i >= n) {   // reported; the pair kernel skips the entry
    if (tid == 0) atomicCAS(err, 0, 1);
    return;
  }
  int a = leaf_of[i];
  // the root is a leaf (D only), or the leaf's parent was left uncompressed
  // (its couplings are dense blocks; the leaf has no basis)
  if (nodes[a].parent < 0 || nodes[nodes[a].parent].state != HSS_COMPRESSED) return;
  double* base = (side ? Vcol : Wrow) + (long long)r * lp1 * kcap;
  {
    const EntryNode& t = nodes[a];
    const int k = side ? t.kc : t.kr;
    const double* X = side ? t.Xc : t.Xr;
    const int pos = (side ? t.ipivc : t.ipivr)[i - t.lo];
    if (pos < 0 || pos >= t.size) {   // not a permutation (never from a compression)
      if (tid == 0) atomicCAS(err, 0, 2);
      return;
    }
    for (int c = tid; c < k; c += 32 * EW) u[c] = pos < k ? (c == pos ? 1.0 : 0.0) : X[c + (long long)(pos - k) * k];
  }
  for (;;) {
    __syncthreads();   // u
    const EntryNode& t = nodes[a];
    const EntryNode& p = nodes[t.parent];
    if (p.state != HSS_COMPRESSED) break;   // dense coupling above: no basis rows needed
    const int ka = side ? t.kc : t.kr, first = p.ch0 == a;
    const EntryNode& b = nodes[first ? p.ch1 : p.ch0];
    double* dst = base + (long long)t.level * kcap;
    // the rows of U_p for the up-step: positions of a's rows in p's pivot order
    const bool top = p.parent < 0;   // a is a child of the root
    const int kp = side ? p.kc : p.kr, mp = side ? p.mc : p.mr;
    const int* inv = top ? nullptr : (side ? p.ipivc : p.ipivr) + (first ? 0 : (side ? b.kc : b.kr));
    auto checked = [&](int q) {
      const int pos = inv[q];
      return pos < 0 || pos >= mp ? -1 : pos;   // (not a permutation: never from a compression)
    };
    auto place = [&](int q) { return HAVE_SP ? sp[q] : checked(q); };
    if (!top) {
      for (int q = tid; q < ka; q += 32 * EW) {
        const int pos = checked(q);
        if (pos < 0) atomicCAS(err, 0, 2);
        if (HAVE_SP) sp[q] = pos;
      }
      for (int c = tid; c < kp; c += 32 * EW) u2[c] = 0.0;
    }
    if (side == 0) {
      // W = u_a(i) B_ab: B12 is kr(nu1) x kc(nu2) with ld max(kr(nu1), 1),
      // B21 is kr(nu2) x kc(nu1) with ld max(kr(nu2), 1)
      const double* B = first ? p.B12 : p.B21;
      const int ld = max(ka, 1), nb = b.kc;
      for (int c0 = 8 * warp; c0 < nb; c0 += 8 * EW) {
        double acc[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) acc[x] = 0.0;
        for (int q = lane; q < ka; q += 32) {
          const double uq = u[q];
          const double* col = B + q + (long long)c0 * ld;
          double m[8];
#pragma unroll
          for (int x = 0; x < 8; ++x) m[x] = c0 + x < nb ? col[(long long)x * ld] : 0.0;
#pragma unroll
          for (int x = 0; x < 8; ++x) acc[x] = __fma_rn(uq, m[x], acc[x]);
        }
        const double s = warp_sum8(acc, lane);
        if ((lane & 3) == 0 && c0 + lane / 4 < nb) dst[c0 + lane / 4] = s;
      }
    } else {
      for (int c = tid; c < ka; c += 32 * EW) dst[c] = u[c];
    }
    if (top) break;
    __syncthreads();   // sp, u2
    // u_parent(i) = u_a(i) U_p(off + q, :), U_p(s, c) = [pos_s == c] for the
    // skeleton rows, X_p(c, pos_s - k_p) for the others
    const double* X = side ? p.Xc : p.Xr;
    for (int c0 = 32 * warp; c0 < kp; c0 += 32 * EW) {
      const int c = c0 + lane;
      double s = 0.0;
      for (int q0 = 0; q0 < ka; q0 += 8) {
        double m[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) {
          const int pos = q0 + x < ka ? place(q0 + x) : -1;
          m[x] = pos >= kp && c < kp ? X[c + (long long)(pos - kp) * kp] : 0.0;
        }
#pragma unroll
        for (int x = 0; x < 8; ++x)
          if (q0 + x < ka && place(q0 + x) >= kp) s = __fma_rn(u[q0 + x], m[x], s);
      }
      if (c < kp) u2[c] = s;
    }
    __syncthreads();
    for (int q = tid; q < ka; q += 32 * EW)   // the skeleton rows: each position once
      if (const int pos = place(q); pos >= 0 && pos < kp) u2[pos] += u[q];
    double* tmp = u;
    u = u2;
    u2 = tmp;
    a = t.parent;
  }
}

// out(r, c) = H(I[r], J[c]) for one chunk of rows and columns: a warp takes
// eight rows of one column, lanes along the dot products (a thread per entry
// walked 64 cache lines per step of a warp).
__global__ void __launch_bounds__(128) k_entry_pairs(const EntryNode* __restrict__ nodes, const int* __restrict__ leaf_of,
                                                     int n, const int* __restrict__ I, int nr,
                                                     const int* __restrict__ J, int nc, const double* __restrict__ Wrow,
                                                     const double* __restrict__ Vcol, int kcap, int lp1,
                                                     double* __restrict__ out, long long ldo) {
  const int lane = threadIdx.x % 32, r0 = (blockIdx.x * 4 + threadIdx.x / 32) * 8, c = blockIdx.y;
  if (r0 >= nr || c >= nc) return;
  const int j = J[c];
  // lane l finds the place of entry l / 4: the levels of the two vectors, their
  // length, or the entry itself
  const int rx = r0 + lane / 4;
  int lev = -1, kb = 0;
  double val = 0.0;
  if (rx < nr && j >= 0 && j < n) {
    const int i = I[rx];
    if (i >= 0 && i < n) {
      int a = leaf_of[i], b = leaf_of[j];
      if (a == b) {
        const EntryNode& t = nodes[a];
        val = t.D[(i - t.lo) + (long long)(j - t.lo) * t.size];
      } else {
        while (nodes[a].level > nodes[b].level) a = nodes[a].parent;
        while (nodes[b].level > nodes[a].level) b = nodes[b].parent;
        while (nodes[a].parent != nodes[b].parent) { a = nodes[a].parent; b = nodes[b].parent; }
        const EntryNode& ta = nodes[a];
        const EntryNode& tb = nodes[b];
        const EntryNode& p = nodes[ta.parent];
        if (p.state != HSS_COMPRESSED) {
          const double* F = p.ch0 == a ? p.F12 : p.F21;   // A(I_a, I_b), ld |a|
          val = F[(i - ta.lo) + (long long)(j - tb.lo) * ta.size];
        } else {
          lev = ta.level;   // (a and b are siblings: one level)
          kb = tb.kc;
        }
      }
    }
  }
  double acc[8];
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    acc[x] = 0.0;
    const int lx = __shfl_sync(0xffffffffu, lev, 4 * x), kx = __shfl_sync(0xffffffffu, kb, 4 * x);
    if (lx < 0) continue;
    const double* w = Wrow + ((long long)(r0 + x) * lp1 + lx) * kcap;
    const double* v = Vcol + ((long long)c * lp1 + lx) * kcap;
    for (int q = lane; q < kx; q += 32) acc[x] = __fma_rn(w[q], v[q], acc[x]);
  }
  const double s = warp_sum8(acc, lane);
  if ((lane & 3) == 0 && rx < nr) out[rx + (long long)c * ldo] = lev >= 0 ? s : val;
}

}  // namespace

cudaError_t launch_leaf_of(const EntryNode* nodes, int nn, int* leaf_of, cudaStream_t st) {
  if (nn <= 0) return cudaSuccess;
  k_leaf_of<<<nn, 128, 0, st>>>(nodes, leaf_of);
  return cudaGetLastError();
}

cudaError_t launch_inv_piv(const EntryNode* nodes, int nn, int* err, cudaStream_t st) {
  if (nn <= 0) return cudaSuccess;
  k_inv_piv<<<2 * nn, 256, 0, st>>>(nodes, nn, err);
  return cudaGetLastError();
}

cudaError_t launch_entry_paths(const EntryNode* nodes, const int* leaf_of, int n, const int* I, int nr, const int* J,
                               int nc, double* Wrow, double* Vcol, int kcap, int lp1, int* err, cudaStream_t st) {
  if (nr + nc <= 0) return cudaSuccess;
  const bool have_sp = (sizeof(double) * 2 + sizeof(int)) * (size_t)kcap <= size_t(227) << 10;
  const size_t sm = (sizeof(double) * 2 + (have_sp ? sizeof(int) : 0)) * (size_t)kcap;
  auto* f = have_sp ? k_entry_paths<true> : k_entry_paths<false>;
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  f<<<nr + nc, 32 * path_warps(kcap), sm, st>>>(nodes, leaf_of, n, I, nr, J, Wrow, Vcol, kcap, lp1, err);
  return cudaGetLastError();
}

cudaError_t launch_entry_pairs(const EntryNode* nodes, const int* leaf_of, int n, const int* I, int nr, const int* J,
                               int nc, const double* Wrow, const double* Vcol, int kcap, int lp1, double* out,
                               long long ldo, cudaStream_t st) {
  if (nr <= 0 || nc <= 0) return cudaSuccess;
  k_entry_pairs<<<dim3((nr + 31) / 32, nc), 128, 0, st>>>(nodes, leaf_of, n, I, nr, J, nc, Wrow, Vcol, kcap, lp1, out,
                                                          ldo);
  return cudaGetLastError();
}

}  // namespace hss
