// FP64 products on the tcgen05 tensor cores, exact up to a rounding below
// FP64's own: C(rows_c(i), j) = alpha sum_l A(i,l) B(l,j) + beta C0(i,j) +
// gamma C(rows_c(i), j), the contract of the FP64 tile kernel (k_gemm.cu),
// for the plain form's sampling, merges, reductions, test projections and the
// HSS product.
//
// Why.  The FP64 pipe has 2 FMA per clock and SM (1.26 TFLOP/s); every one of
// these products was bound by it.  Splitting the operands into integers that
// the tensor core multiplies and adds without any rounding (the error-free
// splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012)
// spends 36 FP16 products on one FP64 product, and the FP16 rate is some 1500
// times the FP64 one.
//
// Measured (one GB300, both orientations, digits made in the call): a dense
// n = 6001 by 200 columns 37.3 ms on the FP64 pipe (k_sample_fp64, 0.77
// TFLOP/s, its last wave half empty) -> 1.40 ms; n = 8192 by 1024 columns 7.4
// ms (37 TFLOP/s), of which the product kernel 6.7 ms (41 TFLOP/s, 3750
// clocks per k-tile: near the 3456 in which shared memory can deliver the
// 72 MMA operand pairs), the digits 0.48 and the maxima 0.11 ms (the latter
// two at 4.5 TB/s).  Relative error against 64 bits 5e-17 (one rounding)
// where the FMA chain had 1e-15 to 2.7e-15.
//
// Digits.  With 2^(e-1) <= the largest |A(i, :)| < 2^e, every element of the
// row is a fixed-point number f 2^(e+1-63), |f| < 2^62, rounded once to an
// integer (elements within 2^-9 of the largest are exact; the others carry an
// error of 2^-63 of it).  f + 0x8080808080808080 has bytes b_7 .. b_0 with
// f = sum (b_p - 128) 2^(8 p): eight signed digits, exact in FP16.  The
// columns of B are cut the same way.  With digit s = 0 the leading one, the
// products of digits p and q weigh 2^-8(p+q); those with p + q <= 7 are
// formed (the rest is below 2^-57 of row maximum x column maximum a term, and
// near 2^-60 for digits of either sign).  Digit 0 is at most
// 2^6, the others 2^7, so the products of weight s >= 1 over K terms sum to
// at most K s 2^14: exact in the FP32 accumulator for K up to 128.
//
// Accumulation.  One TMEM buffer of 64 columns per weight s (8 x 64 = the 512
// columns).  Three warps issue the MMAs of a k-tile side by side, each the
// twelve digit pairs of its own weights in turn, so that neighbouring MMAs add
// into different buffers (one warp that finished weight after weight took
// 12000 clocks per k-tile, three 5800, three alternating 3750).  Sixteen warps
// drain a chain of four k-tiles (128 products of each pair: below 2^24, exact)
// and add every weight at its place into one of two 64-bit sums, (s = 0..3)
// and (s = 4..7), exact for K up to 2^22.  So the whole sum is exact, its order
// does not matter (K can be split over CTAs with integer atomics and the
// result is the same bit for bit), and the only roundings are those of the
// operands' tails and one to FP64 at the end, done in integer arithmetic.
//
// Tile.  128 x 64: the sums take 64 of the 96 registers that twenty warps can
// have, and 96 KB of digits per k-tile leave two stages in shared memory.
//
// What the digits cannot hold: NaN and Inf, and a column of B whose elements
// are of uneven magnitude (fewer than 15/16 of them within 2^-10 of the
// largest).  Such a tile is computed with FP64 FMAs.
//
// What they do not settle.  The scales are those of whole rows and columns, so
// an element of C keeps FP64's accuracy only if its own terms are not all small
// against them: a row whose one large entry meets a zero of B has only terms
// that were cut (with the row (1, 1e-20, ...) all of them).  In units of f, the
// pairs left out are at most 7.03 2^62 a term and the operands' roundings 2^62,
// together 2^65.01: K 2^65.01 in all.  FP64 FMAs guarantee K 2^-53 S, S = sum
// |A(i,l) B(l,j)|, and the digits no less where S >= 2^118 (in f), a
// 1/16 to 1/64 of (largest of the row) x (largest of the column).  k_xs_check
// forms a lower bound of S for every element from the two leading digits, an
// FP16 product that stops as soon as all elements of its tile have reached it
// (for even data after the first 32 of K); elements that never do are computed
// with FP64 FMAs, or, if they are more than one in eight, the whole tile.
//
// A wait that runs out (2 s) loses no result: the tile's last CTA, once its own
// copies and products are over, computes it with FP64 FMAs.  Calls that return
// a status after their work also report the wait (err).
#include <cuda_fp16.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "tc_common.cuh"

namespace hss {
namespace {

constexpr int XD = 8;                                   // digits
constexpr int XKC = XS_BK / 8;                          // 16-byte chunks of 8 FP16 per row
constexpr uint32_t XA = (uint32_t)XS_TM * XS_BK * 2;    // bytes of one digit's tile of A
constexpr uint32_t XB = (uint32_t)XS_TN * XS_BK * 2;    // and of B
constexpr uint32_t XSTAGE = XD * (XA + XB);
constexpr int XNS = 2;                                  // stages (192 KB)
constexpr int XW = 16;                                  // drain warps
constexpr int XMW = 3;                                  // warps that issue MMAs
constexpr int XTHREADS = (1 + XMW + XW) * 32;
constexpr int XNH = XS_TN / 4;                          // columns per drain thread
constexpr int MAXK = 128, MAXR = 32;                    // one maxima unit: k range, rows
constexpr unsigned HI_INF = 0x7FF00000u;
constexpr uint32_t MAGIC = 0x4B400000u;                 // bits of 1.5 2^23

__device__ __forceinline__ const double* op_row(const Opnd& o, int i) {
  int r = o.rows ? o.rows[i] : i;
  const double* b = o.p;
  if (r >= o.split) { b = o.p2; r -= o.split; }
  return b + (long long)r * o.rs;
}

// key of an element's magnitude: the high word without its sign, at least 1
// for a nonzero element
__device__ __forceinline__ unsigned mag_key(double x) {
  return ((unsigned)__double2hiint(x) & 0x7FFFFFFFu) | (__double2loint(x) != 0 ? 1u : 0u);
}

// biased exponent of a row's scale (subnormal rows use the smallest normal)
__device__ __forceinline__ int scale_exp(unsigned key) { return max((int)(key >> 20), 1); }

// f + 0x80..80 of the digits: f = rint(x 2^(63 - E)), E = eM - 1023 + 2 for
// the biased scale exponent eM >= x's own
__device__ __forceinline__ unsigned long long digits8(double x, int eM) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(u >> 52) & 0x7FF;
  unsigned long long m = u & 0xFFFFFFFFFFFFFull;
  if (e) m |= 1ull << 52;
  m <<= 9;
  const int sh = eM - max(e, 1);
  unsigned long long f = sh > 62 ? 0ull : (m + ((1ull << sh) >> 1)) >> sh;
  if ((long long)u < 0) f = 0ull - f;
  return f + 0x8080808080808080ull;
}

// Eight consecutive elements along K: their digits as eight chunks of 16 bytes
// (digit s = byte 7 - s).  0x6400 | b is the FP16 number 1024 + b.
__device__ __forceinline__ void store_digits(uint8_t* dst, uint32_t digit_bytes, const double* v, int eM) {
  uint32_t lo[8], hi[8];
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    const unsigned long long f = digits8(v[x], eM);
    lo[x] = (uint32_t)f;
    hi[x] = (uint32_t)(f >> 32);
  }
  const __half2 off = __half2half2(__ushort_as_half((unsigned short)0x6480));   // 1152
#pragma unroll
  for (int s = 0; s < XD; ++s) {
    const int byte = 7 - s;
    uint32_t w[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const uint32_t a = byte >= 4 ? hi[2 * x] : lo[2 * x], b = byte >= 4 ? hi[2 * x + 1] : lo[2 * x + 1];
      const uint32_t pair = __byte_perm(a, b, (unsigned)(byte & 3) | ((unsigned)((byte & 3) + 4) << 8));   // bytes (a, ., b, .)
      const uint32_t h = __byte_perm(pair, 0x64646464u, 0x4240);   // a, 0x64, b, 0x64
      const __half2 d = __hsub2(*(const __half2*)&h, off);
      w[x] = *(const uint32_t*)&d;
    }
    *(uint4*)(dst + s * digit_bytes) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// offset of chunk c of row r in one digit's tile (canonical K-major layout,
// 4 chunks per row: core matrices of 8 rows x 16 B)
__device__ __forceinline__ uint32_t chunk_off(int r, int c) {
  return (uint32_t)(r / 8) * 512u + (uint32_t)c * 128u + (uint32_t)(r % 8) * 16u;
}

// job of unit u: prefix[j] <= u < prefix[j + 1]
__device__ __forceinline__ int find_job(const int* prefix, int njobs, int u) {
  int lo = 0, hi = njobs;
  while (hi - lo > 1) {
    const int mid = (lo + hi) / 2;
    if (prefix[mid] <= u) lo = mid;
    else hi = mid;
  }
  return lo;
}

// ------------------------------------------------------------ operand maxima
// One unit: 32 rows of A (or columns of B) x 128 of K; one read of the operand.
// A warp takes four rows, all their loads in flight together (with 128 rows to
// a unit, a warp's sixteen rows one after the other took 25 us whatever the
// size).
__global__ void __launch_bounds__(256) k_xs_max(const GemmJob* __restrict__ jobs, const int* __restrict__ prefix,
                                                int njobs) {
  const int ji = find_job(prefix, njobs, blockIdx.x);
  const GemmJob& j = jobs[ji];
  int u = blockIdx.x - prefix[ji];
  const int nkc = (j.K + MAXK - 1) / MAXK, nrb = (j.M + MAXR - 1) / MAXR;
  const int which = u >= nrb * nkc;
  if (which) u -= nrb * nkc;
  const int r0 = (u / nkc) * MAXR, l0 = (u % nkc) * MAXK, l1 = min(j.K, l0 + MAXK);
  const int nr = min(which ? j.N : j.M, r0 + MAXR) - r0;
  const Opnd& o = which ? j.B : j.A;
  unsigned* out = (which ? j.eb : j.ea) + r0;
  const bool rows_fast = which ? o.cs == 1 : (o.rs == 1 && !o.rows);
  const long long cs = o.cs;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  auto at = [&](int r, int l) {
    return which ? op_row(o, l)[(long long)(r0 + r) * cs] : op_row(o, r0 + r)[(long long)l * cs];
  };
  if (rows_fast) {   // lanes along the rows, a warp every eighth l
    unsigned k = 0u;
    if (lane < nr)
      for (int lb = l0 + warp; lb < l1; lb += 64) {
        double v[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) v[x] = lb + 8 * x < l1 ? at(lane, lb + 8 * x) : 0.0;
#pragma unroll
        for (int x = 0; x < 8; ++x) k = max(k, mag_key(v[x]));
      }
    if (k) atomicMax(out + lane, k);
  } else {   // lanes along l
    unsigned k[4] = {0u, 0u, 0u, 0u};
    for (int lb = l0 + lane; lb < l1; lb += 64) {
      double v[4][2];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int x = 0; x < 2; ++x)
          v[q][x] = 4 * warp + q < nr && lb + 32 * x < l1 ? at(4 * warp + q, lb + 32 * x) : 0.0;
#pragma unroll
      for (int q = 0; q < 4; ++q) k[q] = max(k[q], max(mag_key(v[q][0]), mag_key(v[q][1])));
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const unsigned m = __reduce_max_sync(0xffffffffu, k[q]);
      if (lane == 0 && m) atomicMax(out + 4 * warp + q, m);
    }
  }
}

// ----------------------------------------------------------------- digits
// One unit: one k-tile of 128 rows of A or 64 columns of B.  Written once
// per operand element (16 bytes for its 8), read by every tile that uses it.
__global__ void __launch_bounds__(256) k_xs_pack(const GemmJob* __restrict__ jobs, const int* __restrict__ prefix,
                                                 int njobs) {
  __shared__ unsigned s_near[XS_TN];
  const int ji = find_job(prefix, njobs, blockIdx.x);
  const GemmJob& j = jobs[ji];
  int u = blockIdx.x - prefix[ji];
  const int nrb = (j.M + XS_TM - 1) / XS_TM, K = j.K, tid = threadIdx.x;
  const int which = u >= nrb * j.nkt;
  if (which) u -= nrb * j.nkt;
  const int tile = u / j.nkt, kt = u % j.nkt, k0 = kt * XS_BK;
  if (!which) {
    uint8_t* dst = j.pa + ((size_t)tile * j.nkt + kt) * (XD * (size_t)XA);
    const int i0 = tile * XS_TM;
    const bool rows_fast = j.A.rs == 1 && !j.A.rows;
    const long long cs = j.A.cs;
    for (int q = tid; q < XS_TM * XKC; q += 256) {
      const int r = rows_fast ? q % XS_TM : (q / (8 * XKC)) * 8 + (q % 8), c = rows_fast ? q / XS_TM : (q / 8) % XKC;
      const int i = i0 + r;
      const double* row = i < j.M ? op_row(j.A, i) : nullptr;
      double v[8];
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        const int l = k0 + c * 8 + x;
        v[x] = (row && l < K) ? row[(long long)l * cs] : 0.0;
      }
      store_digits(dst + chunk_off(r, c), XA, v, scale_exp(row ? j.ea[i] : 0u));
    }
  } else {
    if (tid < XS_TN) s_near[tid] = 0u;
    __syncthreads();
    uint8_t* dst = j.pb + ((size_t)tile * j.nkt + kt) * (XD * (size_t)XB);
    const int j0 = tile * XS_TN;
    const bool rows_fast = j.B.cs == 1;
    const long long cs = j.B.cs;
    const int q = tid;   // 64 x 4 chunks = 256
    const int r = rows_fast ? q % XS_TN : (q / (8 * XKC)) * 8 + (q % 8), c = rows_fast ? q / XS_TN : (q / 8) % XKC;
    const int col = j0 + r;
    const unsigned key = col < j.N ? j.eb[col] : 0u;
    const int eM = scale_exp(key);
    double v[8];
    unsigned near = 0u;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      const int l = k0 + c * 8 + x;
      v[x] = (col < j.N && l < K) ? op_row(j.B, l)[(long long)col * cs] : 0.0;
      const unsigned mk = mag_key(v[x]);
      near += (mk != 0u && (int)(mk >> 20) + 10 >= eM) ? 1u : 0u;
    }
    store_digits(dst + chunk_off(r, c), XB, v, eM);
    atomicAdd(&s_near[r], near);
    __syncthreads();
    if (tid < XS_TN && j0 + tid < j.N) atomicAdd(j.nb + j0 + tid, s_near[tid]);
  }
}

// ------------------------------------------------- the sampling's operand A
// No leaf holds both a row of [r0, r0 + nr) and a column of [k0, k0 + nk): a
// leaf is a range of indices, so one that holds both holds the ends of the
// two ranges that face each other (its number says nothing about its place:
// the leaves of an uneven tree are numbered level by level).
__device__ __forceinline__ bool tile_clean(const int* leaf_id, int n, int r0, int nr, int k0, int nk) {
  const int r1 = min(r0 + nr, n), k1 = min(k0 + nk, n);
  if (r1 <= k0) return k0 >= n || leaf_id[r1 - 1] != leaf_id[k0];
  if (k1 <= r0) return r0 >= n || leaf_id[k1 - 1] != leaf_id[r0];
  return false;
}

// Largest entry of every row of A - D^(L) and, from the same read, of every
// column (out_t).  A CTA takes 128 rows x 128 columns.  The point kernels
// decrease with the distance, so their largest entry is that of the smallest
// distance (no exponential, root or division per pair).
__global__ void __launch_bounds__(256) k_xs_src_max(SrcDev src, unsigned* out, unsigned* out_t) {
  __shared__ unsigned s_row[128], s_col[128];
  const int n = src.n, tid = threadIdx.x, r = tid % 128, g = tid / 128;
  const int i = blockIdx.x * 128 + r, k0 = blockIdx.y * 128;
  if (tid < 128) { s_row[tid] = 0u; s_col[tid] = 0u; }
  __syncthreads();
  const int li = i < n ? src.leaf_id[i] : -1;
  unsigned km = 0u;
  if (src.kind == HSS_SRC_GAUSS || src.kind == HSS_SRC_LAPLACE) {
    double best = 1.0 / 0.0;
    bool any = false, nan = false;
    const int dim = src.kind == HSS_SRC_GAUSS ? src.dim : 3;
    if (i < n)
      for (int k = k0 + g; k < min(n, k0 + 128); k += 2) {
        if (src.leaf_id[k] == li) continue;
        double r2 = 0.0;
        for (int c = 0; c < dim; ++c) {
          const double t = src.a[i + c * src.ld] - src.a[k + c * src.ld];
          r2 = __fma_rn(t, t, r2);
        }
        any = true;
        if (!(r2 >= 0.0)) nan = true;
        if (r2 < best) best = r2;
      }
    if (any) {
      // the formulas of entry() at the smallest distance; exp is within an ulp but
      // not promised to be monotone, so the entry at a larger distance may be a
      // little above it (and in the next binade, for which the digits have no room)
      const double v = src.kind == HSS_SRC_GAUSS ? exp(-best / (2.0 * src.p0 * src.p0)) * (1.0 + 0x1p-50)
                                                 : 1.0 / (4.0 * 3.141592653589793 * sqrt(best));
      km = nan ? HI_INF : mag_key(v);
    }
    if (km) atomicMax(&s_row[r], km);
  } else {
    // k is uniform over the warp; no leaf of the rows reaches the columns in
    // most tiles
    const bool clean = tile_clean(src.leaf_id, n, blockIdx.x * 128, 128, k0, 128);
    constexpr int UN = 16;   // loads in flight per thread
    for (int kb = k0 + g; kb < min(n, k0 + 128); kb += 2 * UN) {
      double v[UN];
#pragma unroll
      for (int x = 0; x < UN; ++x) {
        const int k = kb + 2 * x;
        v[x] = i < n && k < n && (clean || src.leaf_id[k] != li) ? entry(src, i, k) : 0.0;
      }
#pragma unroll
      for (int x = 0; x < UN; ++x) {
        unsigned key = mag_key(v[x]);
        km = max(km, key);
        if (out_t) {
          key = __reduce_max_sync(0xffffffffu, key);
          if ((tid & 31) == 0 && key) atomicMax(&s_col[kb + 2 * x - k0], key);
        }
      }
    }
    if (km) atomicMax(&s_row[r], km);
  }
  __syncthreads();
  if (tid < 128) {
    if (i < n && s_row[tid]) atomicMax(out + i, s_row[tid]);
  } else if (out_t) {
    const int k = k0 + tid - 128;
    if (k < n && s_col[tid - 128]) atomicMax(out_t + k, s_col[tid - 128]);
  }
}

// The digits of one 128 x 32 tile of A - D^(L) (TRANS: of its transpose).
template <int TRANS>
__global__ void __launch_bounds__(256) k_xs_src_pack(SrcDev src, int row0, int nkt, const unsigned* __restrict__ ea,
                                                     uint8_t* out) {
  const int n = src.n;
  const int rb = blockIdx.x / nkt, kt = blockIdx.x % nkt, k0 = kt * XS_BK;
  uint8_t* dst = out + (size_t)blockIdx.x * (XD * (size_t)XA);
  const bool clean = tile_clean(src.leaf_id, n, row0 + rb * XS_TM, XS_TM, k0, XS_BK);
  for (int q = threadIdx.x; q < XS_TM * XKC; q += 256) {
    const int r = TRANS ? (q / (8 * XKC)) * 8 + (q % 8) : q % XS_TM, c = TRANS ? (q / 8) % XKC : q / XS_TM;
    const int i = row0 + rb * XS_TM + r;
    const int li = i < n && !clean ? src.leaf_id[i] : -1;
    double v[8];
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      const int k = k0 + c * 8 + x;
      double e = 0.0;
      if (i < n && k < n && (clean || src.leaf_id[k] != li)) e = TRANS ? entry(src, k, i) : entry(src, i, k);
      v[x] = e;
    }
    store_digits(dst + chunk_off(r, c), XA, v, scale_exp(i < n ? ea[i] : 0u));
  }
}

// ------------------------------------------------------------------ product
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}

__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(p));
  return p != 0u;
}

// The weights of the issuing warps (twelve digit pairs of a k-tile each) and
// the end of their accumulation chains: four k-tiles, staggered so that the
// drain warps read one warp's buffers while the others' products go on.
__device__ __forceinline__ bool chain_end(int g, int it, int nk) { return ((it + g) & 3) == 3 || it == nk - 1; }

// One issuing warp: all digit pairs of the weights S... of every k-tile.  The
// weights alternate, so that neighbouring MMAs add into different buffers.
// The whole warp waits, the elected lane issues.
template <int G, int... S>
__device__ void issue_weights(uint8_t* smem, uint64_t* full, uint64_t* empty, uint64_t* tfull, uint64_t* tempty,
                              uint32_t tmem, uint32_t id, int nk, bool one, int* err) {
  bool first = true;
  uint32_t chain = 0u;
  for (int it = 0; it < nk; ++it) {
    const int st = it % XNS;
    if (first && !mbar_wait_warp(&tempty[G], (chain & 1u) ^ 1u, err, 33)) return;
    if (!mbar_wait_warp(&full[st], (uint32_t)(it / XNS) & 1u, err, 32)) return;
    const uint64_t ad = sdesc(smem_u32(smem + st * XSTAGE), 128u, 512u);
    const uint64_t bd = sdesc(smem_u32(smem + st * XSTAGE + XD * XA), 128u, 512u);
    const bool end = chain_end(G, it, nk);
    tc_fence_after();
    if (one) {
      const uint32_t fresh = first ? 0u : 1u;
#pragma unroll
      for (int p = 0; p < XD; ++p) {
#pragma unroll
        for (int ks = 0; ks < XS_BK / 16; ++ks) {   // 256 bytes = two chunks per MMA
          auto pair = [&](auto sc) {
            constexpr int s = decltype(sc)::value;
            if (p <= s)
              mma_f16(tmem + (uint32_t)(s * XS_TN), ad + (uint64_t)((p * XA + ks * 256u) >> 4),
                      bd + (uint64_t)(((s - p) * XB + ks * 256u) >> 4), id, (p == 0 && ks == 0) ? fresh : 1u);
          };
          (pair(std::integral_constant<int, S>{}), ...);
        }
      }
      mma_commit(&empty[st]);
      if (end) mma_commit(&tfull[G]);
    }
    __syncwarp();
    first = end;
    if (end) ++chain;
  }
}

// Drain warps: add one weight's 16 columns into the sums.  A chain of 128
// products of each pair stays below s 2^21: weights 0 .. 2 hold the integer
// in the low bits of v + 1.5 2^23 (the caller takes the offset off at the
// end), the others are converted.
template <int S>
__device__ __forceinline__ void drain_weight(uint32_t ta, unsigned long long* hi, unsigned long long* lo) {
  float v[XNH];
  tmem_ld16_nw(ta + (uint32_t)(S * XS_TN), v);
  tmem_wait_ld();
#pragma unroll
  for (int x = 0; x < XNH; ++x) {
    unsigned long long& a = S < 4 ? hi[x] : lo[x];
    if constexpr (S <= 2) {
      const uint32_t raw = __float_as_uint(__fadd_rn(v[x], 12582912.0f));
      a += (unsigned long long)raw * (1u << (24 - 8 * (S & 3)));
    } else {
      a += (unsigned long long)((long long)__float2int_rn(v[x]) * (1 << (24 - 8 * (S & 3))));
    }
  }
}
template <int G, int... S>
__device__ __forceinline__ bool drain_weights(uint64_t* tfull, uint64_t* tempty, uint32_t chain, uint32_t ta, int lane,
                                              unsigned long long* hi, unsigned long long* lo, int* err) {
  if (!mbar_wait_warp(&tfull[G], chain & 1u, err, 34)) return false;
  tc_fence_after();
  (drain_weight<S>(ta, hi, lo), ...);
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive(&tempty[G]);
  return true;
}

__device__ __forceinline__ void bar_drain() { asm volatile("bar.sync 1, %0;" ::"n"(XW * 32) : "memory"); }

// (hi 2^32 + lo) 2^e2 rounded once to FP64 (nearest even), negated if neg;
// integer operations (the FP64 conversions run at the rate of the FP64 pipe)
__device__ __forceinline__ double fixed_value(long long hi, long long lo, int e2, bool neg) {
  hi += lo >> 32;
  uint32_t L = (uint32_t)lo;
  if (hi < 0) {
    neg = !neg;
    hi = ~hi;
    L = ~L + 1u;
    if (L == 0u) ++hi;
  }
  unsigned long long top;
  bool sticky = false;
  int ex;
  if (hi) {
    const int lz = __clzll(hi);
    const unsigned long long L64 = (unsigned long long)L << 32;
    top = lz ? ((unsigned long long)hi << lz) | (L64 >> (64 - lz)) : (unsigned long long)hi;
    sticky = (L64 << lz) != 0ull;
    ex = 95 - lz;
  } else {
    if (L == 0u) return 0.0;
    const int lz = __clz(L);
    top = (unsigned long long)L << (32 + lz);
    ex = 31 - lz;
  }
  unsigned long long m = top >> 11;
  const uint32_t rem = (uint32_t)top & 0x7FFu;
  if (rem > 0x400u || (rem == 0x400u && (sticky || (m & 1ull)))) ++m;
  const int E = ex + e2;
  if (E >= -1022 && E <= 1023) {
    const unsigned long long b = ((unsigned long long)(E + 1022) << 52) + m;   // m's leading bit adds 1 to E + 1022
    return __longlong_as_double((long long)(b | (neg ? 1ull << 63 : 0ull)));
  }
  const double v = scalbn((double)m, E - 52);
  return neg ? -v : v;
}

// The tile's results (column-padded, in shared memory) to C: lanes along the
// contiguous direction.
constexpr int XLD = XS_TN + 1;
__device__ __forceinline__ void store_one(const GemmJob& jb, int i, int jj, double v) {
  if (jb.beta != 0.0) {
    const double c0 = op_row(jb.C0, i)[(long long)jj * jb.C0.cs];
    v += jb.beta == 1.0 ? c0 : jb.beta * c0;
  }
  int r = jb.c_rows ? jb.c_rows[i] : i;
  double* base = jb.C;
  if (r >= jb.c_split) { base = jb.C2; r -= jb.c_split; }
  const long long off = (long long)r * jb.c_rs + (long long)jj * jb.c_cs;
  if (jb.gamma != 0.0) v += jb.gamma == 1.0 ? base[off] : jb.gamma * base[off];
  base[off] = v;
  if (jb.dup) jb.dup[off] = v;
}
// (mask: elements to leave out, or NULL)
template <int NR = XS_TM>
__device__ __forceinline__ void store_tile(const GemmJob& jb, const double* sm, int i0, int j0, int t,
                                           const unsigned* mask = nullptr) {
  const bool row_major = jb.c_cs == 1;
  for (int q = t; q < NR * XS_TN; q += XW * 32) {
    const int il = row_major ? q / XS_TN : q % NR, jl = row_major ? q % XS_TN : q / NR;
    const int i = i0 + il, jj = j0 + jl;
    if (i >= jb.M || jj >= jb.N) continue;
    if (mask && (mask[2 * il + jl / 32] >> (jl % 32) & 1u)) continue;
    store_one(jb, i, jj, sm[il * XLD + jl]);
  }
}

// NR rows of the tile by FP64 FMAs (operands the digits cannot hold): 512
// threads, RX x CY outputs each, K staged 16 at a time, every output one chain
// over K whatever NR.
template <int RX, int CY>
__device__ void fp64_rows(const GemmJob& jb, double* sm, int i0, int j0, int t, const unsigned* mask) {
  constexpr int TX = XS_TN / CY, NR = XW * 32 / TX * RX;
  double* stage = sm + XS_TM * XLD;
  double (*As)[NR + 2] = (double (*)[NR + 2])stage;
  double (*Bs)[XS_TN + 2] = (double (*)[XS_TN + 2])(stage + 16 * (NR + 2));
  const int tx = t % TX, ty = t / TX;
  double acc[RX][CY];
#pragma unroll
  for (int a = 0; a < RX; ++a)
#pragma unroll
    for (int b = 0; b < CY; ++b) acc[a][b] = 0.0;
  for (int l0 = 0; l0 < jb.K; l0 += 16) {
    for (int q = t; q < 16 * NR; q += XW * 32) {
      const int il = q % NR, kk = q / NR, i = i0 + il, l = l0 + kk;
      As[kk][il] = (i < jb.M && l < jb.K) ? op_row(jb.A, i)[(long long)l * jb.A.cs] : 0.0;
    }
    for (int q = t; q < 16 * XS_TN; q += XW * 32) {
      const int jl = q % XS_TN, kk = q / XS_TN, jj = j0 + jl, l = l0 + kk;
      Bs[kk][jl] = (jj < jb.N && l < jb.K) ? op_row(jb.B, l)[(long long)jj * jb.B.cs] : 0.0;
    }
    bar_drain();
#pragma unroll 4
    for (int kk = 0; kk < 16; ++kk) {
      double a[RX], b[CY];
#pragma unroll
      for (int x = 0; x < RX; ++x) a[x] = As[kk][ty * RX + x];
#pragma unroll
      for (int x = 0; x < CY; ++x) b[x] = Bs[kk][tx * CY + x];
#pragma unroll
      for (int x = 0; x < RX; ++x)
#pragma unroll
        for (int y = 0; y < CY; ++y) acc[x][y] = __fma_rn(a[x], b[y], acc[x][y]);
    }
    bar_drain();
  }
#pragma unroll
  for (int x = 0; x < RX; ++x)
#pragma unroll
    for (int y = 0; y < CY; ++y) sm[(ty * RX + x) * XLD + tx * CY + y] = jb.alpha * acc[x][y];
  bar_drain();
  store_tile<NR>(jb, sm, i0, j0, t, mask);
}

// Such a tile is shared by its CTAs by rows: those of its K segments, and
// helpers (CTAs past the last unit, which leave at once when the digits hold
// the tile).  One CTA takes 2.15 us per unit of K for the tile, and a level of
// a deep tree has a dozen to fifty tiles: the projections of the Incrementing
// strategy on the surface kernel (n = 4001), where the elements of one
// column spread over more than 2^10, took 300 to 1500 us a product on 12 to 48
// CTAs: 21.1 ms of 77 in all, 6.6 with the rows shared.
// (mask: see store_tile; with one part only)
__device__ __noinline__ void fp64_share(const GemmJob& jb, double* sm, int i0, int j0, int part, int parts, int t,
                                        const unsigned* mask = nullptr) {
  const int ns = parts >= 8 ? 8 : (parts >= 4 ? 4 : (parts >= 2 ? 2 : 1));
  const int r0 = i0 + part * (XS_TM / ns);
  if (part >= ns || r0 >= jb.M) return;
  if (ns == 8) fp64_rows<1, 2>(jb, sm, r0, j0, t, nullptr);
  else if (ns == 4) fp64_rows<1, 4>(jb, sm, r0, j0, t, nullptr);
  else if (ns == 2) fp64_rows<2, 4>(jb, sm, r0, j0, t, nullptr);
  else fp64_rows<4, 4>(jb, sm, r0, j0, t, mask);
}

// The marked elements of every nseg-th row of the tile by FP64 FMAs: a warp an
// element, its lanes along K.
__device__ __noinline__ void fix_rows(const GemmJob& jb, const unsigned* mask, int i0, int j0, int seg, int warp, int lane) {
  for (int q = warp; seg + q * jb.nseg < XS_TM; q += XW) {
    const int il = seg + q * jb.nseg, i = i0 + il;
    if (i >= jb.M) return;
    const double* a = op_row(jb.A, i);
    for (int h = 0; h < 2; ++h) {
      for (unsigned m = mask[2 * il + h]; m; m &= m - 1u) {   // (none past N)
        const int jj = j0 + 32 * h + __ffs(m) - 1;
        double v = 0.0;
#pragma unroll 4
        for (int l = lane; l < jb.K; l += 32)
          v = __fma_rn(a[(long long)l * jb.A.cs], op_row(jb.B, l)[(long long)jj * jb.B.cs], v);
#pragma unroll
        for (int o = 16; o; o /= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) store_one(jb, i, jj, jb.alpha * v);
      }
    }
  }
}

__global__ void __maxnreg__(96) k_xs_mm(const GemmJob* __restrict__ jobs, const int* __restrict__ prefix, int njobs,
                                          int nunits, int leave, int* err) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ GemmJob sj;
  __shared__ int s_last, s_fail, s_redo;
  uint64_t* full = (uint64_t*)(smem + XNS * XSTAGE);
  uint64_t* empty = full + XNS;
  uint64_t* tfull = empty + XNS;    // one per issuing warp
  uint64_t* tempty = tfull + XMW;
  uint64_t* idle = tempty + XMW;    // one per issuing warp: its last product is done
  uint32_t* tmem_slot = (uint32_t*)(idle + XMW);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  // CTAs past the units are helpers of unit blockIdx.x % nunits
  const int share = blockIdx.x / nunits, shares = gridDim.x / nunits, unit = blockIdx.x % nunits;
  const int ji = find_job(prefix, njobs, unit);
  if (tid == 0) {
    sj = jobs[ji];
    s_fail = s_redo = 0;
    for (int s = 0; s < XNS; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], XMW); }
    for (int s = 0; s < XMW; ++s) { mbar_init(&tfull[s], 1); mbar_init(&tempty[s], XW); mbar_init(&idle[s], 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const int u = unit - prefix[ji], nseg = sj.nseg;
  const int ntn = (sj.N + XS_TN - 1) / XS_TN;
  const int t = u / nseg, seg = u % nseg;   // column tiles fastest: the tiles of one row block share A through L2
  const int ti = t / ntn, tj = t % ntn, i0 = ti * XS_TM, j0 = tj * XS_TN;
  const unsigned state = sj.state[t];
  double* tile_sm = (double*)smem;   // the results, once the stages are done with
  if (state & XS_FMA) {
    if (!leave && warp > XMW)
      fp64_share(sj, tile_sm, i0, j0, seg + nseg * share, nseg * shares, tid - (1 + XMW) * 32);
    return;
  }
  if (share > 0) return;
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int kt0 = (int)((long long)sj.nkt * seg / nseg), nk = (int)((long long)sj.nkt * (seg + 1) / nseg) - kt0;
  if (warp == 0) {
    if (lane == 0) {
      const uint8_t* gA = sj.pa + ((size_t)ti * sj.nkt + kt0) * (XD * (size_t)XA);
      const uint8_t* gB = sj.pb + ((size_t)tj * sj.nkt + kt0) * (XD * (size_t)XB);
      int it = 0;
      for (; it < nk; ++it) {
        const int st = it % XNS;
        if (!mbar_wait(&empty[st], ((uint32_t)(it / XNS) & 1u) ^ 1u, err, 31)) break;
        uint8_t* sp = smem + st * XSTAGE;
        mbar_expect_tx(&full[st], XSTAGE);
        bulk_g2s(sp, gA + (size_t)it * (XD * XA), XD * XA, &full[st]);
        bulk_g2s(sp + XD * XA, gB + (size_t)it * (XD * XB), XD * XB, &full[st]);
      }
      // (no copy is under way when this CTA goes on, whatever the others gave up)
      for (int c = max(0, it - XNS); c < it; ++c) mbar_wait(&full[c % XNS], (uint32_t)(c / XNS) & 1u, err, 35);
    }
  } else if (warp <= XMW) {
    const uint32_t id = idesc(0u, (uint32_t)XS_TN);   // FP16 operands
    const bool one = elect_one();
    if (warp == 1) issue_weights<0, 7, 3>(smem, full, empty, tfull, tempty, tmem, id, nk, one, err);
    else if (warp == 2) issue_weights<1, 6, 4>(smem, full, empty, tfull, tempty, tmem, id, nk, one, err);
    else issue_weights<2, 5, 2, 1, 0>(smem, full, empty, tfull, tempty, tmem, id, nk, one, err);
    if (one) mma_commit(&idle[warp - 1]);
    __syncwarp();
    mbar_wait_warp(&idle[warp - 1], 0u, err, 36);
  } else {
    const int q = warp % 4, h = (warp - 1 - XMW) / 4, t512 = tid - (1 + XMW) * 32;
    unsigned long long hi[XNH], lo[XNH];
#pragma unroll
    for (int x = 0; x < XNH; ++x) { hi[x] = 0ull; lo[x] = 0ull; }
    const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(h * XNH);
    bool ok = true;
    uint32_t c0 = 0u, c1 = 0u, c2 = 0u;   // chains drained of each issuing warp
    for (int it = 0; it < nk && ok; ++it) {
      if (ok && chain_end(0, it, nk)) ok = drain_weights<0, 7, 3>(tfull, tempty, c0++, ta, lane, hi, lo, err);
      if (ok && chain_end(1, it, nk)) ok = drain_weights<1, 6, 4>(tfull, tempty, c1++, ta, lane, hi, lo, err);
      if (ok && chain_end(2, it, nk)) ok = drain_weights<2, 5, 2, 1, 0>(tfull, tempty, c2++, ta, lane, hi, lo, err);
    }
#ifdef HSS_TEST_LOST_WAIT   // tests: as if the waits of every other tile's last segment had run out
    if ((t & 1) && seg == nseg - 1) {
      ok = false;
      if (lane == 0) atomicCAS(err, 0, 99);
    }
#endif
    // the offset of the raw values of weights 0 .. 2, once per chain
    const unsigned long long bias = (unsigned long long)MAGIC * 0x01010100ull * (unsigned long long)c2;
#pragma unroll
    for (int x = 0; x < XNH; ++x) hi[x] -= bias;
    if (!ok && lane == 0) {
      s_fail = 1;
      atomicOr(sj.state + t, XS_WAIT);   // (for the tile's last CTA)
    }
    bool last = true;
    if (nseg > 1) {
      // K is split: exact integer sums in global memory, the last CTA to
      // arrive writes the tile
      unsigned long long* ws = sj.ws + (size_t)t * (2 * XS_TM * XS_TN) + t512;
      if (ok) {
#pragma unroll
        for (int x = 0; x < XNH; ++x) {
          atomicAdd(ws + (2 * x) * (XW * 32), hi[x]);
          atomicAdd(ws + (2 * x + 1) * (XW * 32), lo[x]);
        }
      }
      __threadfence();
      bar_drain();
      if (t512 == 0) {
        s_last = atomicAdd(sj.cnt + t, 1u) == (unsigned)(nseg - 1) ? 1 : 0;
        if (s_last && (atomicOr(sj.state + t, 0u) & XS_WAIT)) s_fail = 1;
      }
      bar_drain();
      last = s_last != 0;
      if (last) {
        __threadfence();
#pragma unroll
        for (int x = 0; x < XNH; ++x) {
          hi[x] = __ldcg(ws + (2 * x) * (XW * 32));
          lo[x] = __ldcg(ws + (2 * x + 1) * (XW * 32));
        }
      }
    }
    const int il = 32 * q + lane, i = i0 + il;
    if (last && ok) {
      const int eA = scale_exp(i < sj.M ? sj.ea[i] : 0u);
      const bool neg = sj.alpha == -1.0;
      const double alpha = neg ? 1.0 : sj.alpha;
#pragma unroll
      for (int x = 0; x < XNH; ++x) {
        const int jl = h * XNH + x, jj = j0 + jl;
        const int eB = scale_exp(jj < sj.N ? sj.eb[jj] : 0u);
        // E_a + E_b - 70 with E = e - 1021
        const double v = fixed_value((long long)hi[x], (long long)lo[x], eA + eB - 2042 - 70, neg);
        tile_sm[il * XLD + jl] = alpha == 1.0 ? v : alpha * v;
      }
    }
    bar_drain();   // (every drain warp is here: unless one gave up, all products and copies are done)
    const unsigned* mask = state & XS_PART ? sj.mask + (size_t)t * (2 * XS_TM) : nullptr;
    if (last && !s_fail) store_tile(sj, tile_sm, i0, j0, t512, mask);
    else if (last && t512 == 0) s_redo = 1;
    if (mask && !leave) fix_rows(sj, mask, i0, j0, seg, warp - 1 - XMW, lane);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
  if (s_redo && warp > XMW) {
    if (leave) {
      if (lane == 0) atomicOr(sj.state + t, XS_FMA);
    } else {
      fp64_share(sj, tile_sm, i0, j0, 0, 1, tid - (1 + XMW) * 32, state & XS_PART ? sj.mask + (size_t)t * (2 * XS_TM) : nullptr);
    }
  }
}

// ------------------------------------------------- what the digits settle
// One CTA per tile.  The magnitude of an element by its two leading digits,
// h = max(|d0 + d1 / 256| - 2^-9, 0) <= |f| 2^-56 up to two roundings to FP16
// (the digits below are at most 1.004 2^-9), so sum h_A h_B, with 64 for the
// 2^118 of S above and 1.5 % for the roundings and the 0.01 of the exponent, is a
// lower bound of S.  One k-tile first, then three at a time, from the tile's own
// place outwards (matrices that decay have their large entries near the
// diagonal).  Bound by the latency of its few loads: 5 to 11 us a launch (dense
// n = 6001, 200 columns: 1.39 to 1.40 ms for the call; a product of 2048 columns
// with twelve launch sets 3.73 to 3.84).
constexpr int CKT = 3;                                   // most k-tiles a round
constexpr uint32_t CK_SMEM = CKT * (XA + XB);
constexpr int CK_MOST = XS_TM * XS_TN / 8;               // elements to compute one by one
constexpr float CK_ENOUGH = 65.0f;

__device__ __forceinline__ uint32_t lead_mag(uint32_t d0, uint32_t d1) {   // two FP16 digits each
  const __half2 v = __hfma2(*(const __half2*)&d1, __half2half2(__ushort_as_half((unsigned short)0x1C00)),   // 2^-8
                            *(const __half2*)&d0);
  const __half2 h = __hmax2(__hsub2(__habs2(v), __float2half2_rn(0.00197f)), __float2half2_rn(0.0f));
  return *(const uint32_t*)&h;
}

__global__ void __launch_bounds__(256, 5) k_xs_check(const GemmJob* __restrict__ jobs, const int* __restrict__ prefix,
                                                     int njobs, int* err) {
  __shared__ __align__(1024) uint8_t smem[CK_SMEM];
  __shared__ GemmJob sj;
  __shared__ uint64_t bar;
  __shared__ uint32_t s_tmem;
  __shared__ unsigned s_free[2], s_cnt;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  int ji = 0;   // (one round of loads up to 256 jobs; find_job's chain is eight)
  for (int j = tid; j - tid < njobs; j += 256) ji += __syncthreads_count(j < njobs && prefix[j + 1] <= (int)blockIdx.x);
  if (tid == 0) {
    sj = jobs[ji];
    s_cnt = 0u;
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                 "r"((uint32_t)XS_TN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const int t = blockIdx.x - prefix[ji], ntn = (sj.N + XS_TN - 1) / XS_TN;
  const int ti = t / ntn, tj = t % ntn, i0 = ti * XS_TM, j0 = tj * XS_TN;
  const int nkt = sj.nkt, kt0 = (sj.row0 + i0 + XS_TM / 2) / XS_BK % nkt;
  const uint8_t* gA = sj.pa + (size_t)ti * nkt * (XD * (size_t)XA);
  const uint8_t* gB = sj.pb + (size_t)tj * nkt * (XD * (size_t)XB);
  uint4 d[3][2];   // a thread's 16-byte chunks of one k-tile: two of A, one of B, both digits
  auto fetch = [&](int k) {   // kt0, kt0 + 1, kt0 - 1, kt0 + 2, ...
    int kg = kt0 + (k & 1 ? (k + 1) / 2 : -(k / 2));   // (-nkt < . < 2 nkt)
    if (kg >= nkt) kg -= nkt;
    if (kg < 0) kg += nkt;
    const uint8_t* pa = gA + (size_t)kg * (XD * (size_t)XA) + tid * 16;
    const uint8_t* pb = gB + (size_t)kg * (XD * (size_t)XB) + tid * 16;
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      d[0][x] = *(const uint4*)(pa + x * XA);
      d[1][x] = *(const uint4*)(pa + x * XA + 4096);
      d[2][x] = *(const uint4*)(pb + x * XB);
    }
  };
  fetch(0);
  // operands the digits cannot hold; rows and columns of zeros have no terms
  int bad = 0;
  if (tid < XS_TM) {
    bad = i0 + tid < sj.M && sj.ea[i0 + tid] >= HI_INF;
  } else if (tid < XS_TM + XS_TN) {
    const int c = j0 + tid - XS_TM;
    const unsigned key = c < sj.N ? sj.eb[c] : 0u;
    bad = key >= HI_INF || (key != 0u && (unsigned long long)sj.nb[c] * 16ull < 15ull * (unsigned)sj.K);
    const unsigned fr = __ballot_sync(0xffffffffu, key == 0u);
    if (lane == 0) s_free[(tid - XS_TM) / 32] = fr;
  }
  bad = __syncthreads_or(bad);
  const int row = 32 * (warp % 4) + lane, h = warp / 4;   // a thread's row and half of the columns
  const bool row_free = i0 + row >= sj.M || sj.ea[i0 + row] == 0u;
  const unsigned col_free = s_free[h];
  unsigned fail = 0u, rounds = 0u;   // (rounds: products waited for)
  bool ok = true;
  int more = !bad;
  for (int it = 0, done = 0; done < nkt && more; ++it) {
    const int nk = it ? min(CKT, nkt - done) : 1;
    if (it == 1) fetch(done);
    for (int kt = 0; kt < nk; ++kt) {
#pragma unroll
      for (int x = 0; x < 3; ++x)
        *(uint4*)(smem + (x < 2 ? kt * XA + x * 4096u : CKT * XA + kt * XB) + tid * 16u) =
            make_uint4(lead_mag(d[x][0].x, d[x][1].x), lead_mag(d[x][0].y, d[x][1].y),
                       lead_mag(d[x][0].z, d[x][1].z), lead_mag(d[x][0].w, d[x][1].w));
      if (it && done + kt + 1 < nkt) fetch(done + kt + 1);   // (for the next round, too, while this one is multiplied)
    }
    fence_async_smem();
    __syncthreads();
    if (warp == 0) {
      if (elect_one()) {
        tc_fence_after();
        const uint32_t id = idesc(0u, (uint32_t)XS_TN);
        for (int kt = 0; kt < nk; ++kt) {
          const uint64_t ad = sdesc(smem_u32(smem + kt * XA), 128u, 512u);
          const uint64_t bd = sdesc(smem_u32(smem + CKT * XA + kt * XB), 128u, 512u);
#pragma unroll
          for (int ks = 0; ks < XS_BK / 16; ++ks)
            mma_f16(tmem, ad + (uint64_t)(ks * 16), bd + (uint64_t)(ks * 16), id, it + kt + ks > 0 ? 1u : 0u);
        }
        mma_commit(&bar);
      }
      __syncwarp();
    }
    ok = mbar_wait_warp(&bar, (uint32_t)it & 1u, err, 37);
    tc_fence_after();
    fail = 0u;
    if (ok) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float v[16];
        tmem_ld16_nw(tmem + ((uint32_t)(32 * (warp % 4)) << 16) + (uint32_t)(32 * h + 16 * c), v);
        tmem_wait_ld();
#pragma unroll
        for (int x = 0; x < 16; ++x) fail |= v[x] >= CK_ENOUGH ? 0u : 1u << (16 * c + x);
      }
      fail = row_free ? 0u : fail & ~col_free;
    }
    tc_fence_before();
    if (__syncthreads_or(!ok)) { ok = false; break; }
    more = __syncthreads_or(fail != 0u);
    done += nk;
    ++rounds;
  }
  if (more && ok) {
    atomicAdd(&s_cnt, (unsigned)__popc(fail));
    sj.mask[(size_t)t * (2 * XS_TM) + 2 * row + h] = fail;
  }
  __syncthreads();
  if (tid == 0 && (bad || !ok || more)) sj.state[t] = !bad && ok && s_cnt <= CK_MOST ? XS_PART : XS_FMA;
  if (warp == 1) {
    if (!ok) mbar_wait_warp(&bar, rounds & 1u, err, 38);   // (the products under way)
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)XS_TN) : "memory");
  }
}

}  // namespace

size_t xs_tile_bytes(int which) { return (size_t)XD * (which ? XB : XA); }

int xs_max_units(int M, int N, int K) {
  return ((M + MAXR - 1) / MAXR + (N + MAXR - 1) / MAXR) * ((K + MAXK - 1) / MAXK);
}
int xs_pack_units(int M, int N, int K) {
  return ((M + XS_TM - 1) / XS_TM + (N + XS_TN - 1) / XS_TN) * ((K + XS_BK - 1) / XS_BK);
}

cudaError_t launch_xs_max(const GemmJob* jobs_dev, const int* prefix_dev, int njobs, int nunits, cudaStream_t st) {
  if (nunits <= 0) return cudaSuccess;
  k_xs_max<<<nunits, 256, 0, st>>>(jobs_dev, prefix_dev, njobs);
  return cudaGetLastError();
}

cudaError_t launch_xs_pack(const GemmJob* jobs_dev, const int* prefix_dev, int njobs, int nunits, cudaStream_t st) {
  if (nunits <= 0) return cudaSuccess;
  k_xs_pack<<<nunits, 256, 0, st>>>(jobs_dev, prefix_dev, njobs);
  return cudaGetLastError();
}

cudaError_t launch_xs_check(const GemmJob* jobs_dev, const int* prefix_dev, int njobs, int ntiles, int* err,
                            cudaStream_t st) {
  if (ntiles <= 0) return cudaSuccess;
  k_xs_check<<<ntiles, 256, 0, st>>>(jobs_dev, prefix_dev, njobs, err);
  return cudaGetLastError();
}

cudaError_t launch_xs_mm(const GemmJob* jobs_dev, const int* prefix_dev, int njobs, int nunits, bool leave, int* err,
                         cudaStream_t st) {
  if (nunits <= 0) return cudaSuccess;
  const size_t sm = (size_t)XNS * XSTAGE + 8 * (2 * XNS + 3 * XMW) + 16;
  cudaError_t e = cudaFuncSetAttribute(k_xs_mm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  // helpers where the units leave SMs idle
  const int shares = leave || nunits > 304 ? 1 : std::min(8, 608 / nunits);
  k_xs_mm<<<nunits * shares, XTHREADS, sm, st>>>(jobs_dev, prefix_dev, njobs, nunits, leave ? 1 : 0, err);
  return cudaGetLastError();
}

cudaError_t launch_xs_src_max(const SrcDev& src, unsigned* out, unsigned* out_t, cudaStream_t st) {
  if (src.kind < HSS_SRC_DENSE || src.kind > HSS_SRC_LAPLACE) return cudaErrorInvalidValue;   // no entries on the device
  if (src.n <= 0) return cudaSuccess;
  const unsigned nb = (unsigned)((src.n + 127) / 128);
  if (nb > 65535u) return cudaErrorInvalidValue;
  k_xs_src_max<<<dim3(nb, nb), 256, 0, st>>>(src, out, out_t);
  return cudaGetLastError();
}

cudaError_t launch_xs_src_pack(const SrcDev& src, int trans, int row0, int rows, const unsigned* ea,
                               unsigned char* out, cudaStream_t st) {
  if (src.kind < HSS_SRC_DENSE || src.kind > HSS_SRC_LAPLACE) return cudaErrorInvalidValue;
  if (rows <= 0) return cudaSuccess;
  const int nkt = (src.n + XS_BK - 1) / XS_BK, nrb = (rows + XS_TM - 1) / XS_TM;
  if ((long long)nkt * nrb > 0x7fffffffLL) return cudaErrorInvalidValue;
  if (trans) k_xs_src_pack<1><<<nkt * nrb, 256, 0, st>>>(src, row0, nkt, ea, out);
  else k_xs_src_pack<0><<<nkt * nrb, 256, 0, st>>>(src, row0, nkt, ea, out);
  return cudaGetLastError();
}

}  // namespace hss
