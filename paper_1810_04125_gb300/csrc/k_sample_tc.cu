// Mixed-precision sampling on the tcgen05 tensor cores:
//     S = (A - D^(L)) R        (orientation 0, S^r)
//     S = (A - D^(L))^T R      (orientation 1, S^c)
// i.e. eq. sample_off_diag at the leaf level with the leaf subtraction folded
// into the tile staging, as in the FP64 kernel.
//
// Precision (the two mixed forms):
//   TF32X2: every entry a of A is rounded once to FP32 and split as
//           a ~= a0 + a1 with a0, a1 TF32 values (22 significant bits);
//           R holds TF32 values exactly; two kind::tf32 products.
//   BF16X3: a ~= a0 + a1 + a2 with BF16 terms (24 significant bits); R holds
//           BF16 values exactly; three kind::f16 (bf16) products.
// Every product of terms is exact in FP32; partial sums are kept short in
// TMEM and carried in float-float registers (see "Accumulation" below).
//
// Three kernels share the tile format: the packed kernel streams an A that was
// split once into canonical tiles (cp.async.bulk into an mbarrier ring); the
// generating kernel computes the entries of a point kernel in its producer
// warps; the Toeplitz kernel reads every tile out of a strip of the few core
// matrices that such tiles are made of.  One thread issues tcgen05.mma, the
// R tile arrives pre-packed by bulk copy, and every mbarrier wait is bounded
// (about 2 s of %globaltimer): on expiry the kernel records an error code,
// leaves its loops, frees its TMEM and returns.
//
// The shared-memory tile layout and the accumulation scheme are described in
// tc_common.cuh.
#include <stdint.h>

#include <algorithm>

#include "tc_common.cuh"

namespace hss {
namespace {

constexpr int NSTAGE = 3;                  // stages of the generating kernel

// Entry A(i, j) for the generating producers.  The Laplace kernel
// 1 / (4 pi |x_i - x_j|) avoids the FP64 square root and division (long
// sequences on the FP64 pipe, which bounds this kernel): |x_i - x_j|^-1 from
// the FP32 reciprocal square root of r^2, refined by one Newton-Raphson step
// for x^(-1/2), y1 = y0 (3 - r^2 y0^2) / 2, in FP64 — relative error about
// 1.5 e0^2 for an initial error e0 ~ 1e-7, far below the split that follows.
// r^2 outside the FP32 normal range, the diagonal and the other kinds take
// the plain definition.
__device__ __forceinline__ double entry_gen(const SrcDev& s, int i, int j) {
  if (s.kind != HSS_SRC_LAPLACE || i == j) return entry(s, i, j);
  double r2 = 0.0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double t = s.a[i + c * s.ld] - s.a[j + c * s.ld];
    r2 = __fma_rn(t, t, r2);
  }
  const float r2f = __double2float_rn(r2);
  if (!(r2f >= 1.1754943508222875e-38f) || !(r2f <= 1e38f)) return entry(s, i, j);
  const double y0 = (double)rsqrtf(r2f);
  const double y1 = y0 * __fma_rn(-0.5 * r2 * y0, y0, 1.5);
  return y1 * (1.0 / (4.0 * 3.141592653589793));
}

// The Laplace entry rounded to FP32, from points split into pairs of floats, on
// the FP32 pipe (64 times the FP64 pipe's rate; entry_gen takes nine FP64
// instructions and four conversions per entry, which bounded the generation).
// The coordinate differences, their squares and the sum are kept as unevaluated
// pairs with error-free additions and products (Dekker, Numer. Math. 18, 1971;
// Knuth, TAOCP 2, 4.2.2), 1/sqrt by one Newton step of third order on the FP32
// reciprocal square root with an exact residual: relative error below 2^-44.
// Returns false, and the caller evaluates entry_gen, where that is not certain
// to give entry_gen's FP32 value, so that the samples are the same bit for bit:
// where the value is closer to a rounding boundary than what the two can differ
// by, 2^-41 of it for the arithmetic of both and 2^-43 max|coordinate| / r for
// the coordinates (split to 2^-48 of themselves, subtracted to 2^-46), or r^2 is
// far from 1 (or not finite).  One entry in 2^15 at max|coordinate| / r = 2.
// About 105 instructions an entry with the split: 2.8 ps at full issue, and the
// pack kernel, which evaluates one half, took 5.8 an entry of the whole.
// n = 12000, 128 columns, BF16 x 3: 6.44 ms with entry_gen, 1.04 ms so.
__device__ __forceinline__ bool laplace_f32(const float4 ah, const float4 al, const float4 bh, const float4 bl,
                                            float* out) {
  float p[3], pe[3];
  const float a1[3] = {ah.x, ah.y, ah.z}, a2[3] = {al.x, al.y, al.z};
  const float b1[3] = {bh.x, bh.y, bh.z}, b2[3] = {bl.x, bl.y, bl.z};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float s = __fsub_rn(a1[c], b1[c]), t = __fsub_rn(s, a1[c]);
    float e = __fsub_rn(__fsub_rn(a1[c], __fsub_rn(s, t)), __fadd_rn(b1[c], t));
    e = __fadd_rn(e, __fsub_rn(a2[c], b2[c]));
    p[c] = __fmul_rn(s, s);
    pe[c] = __fmaf_rn(e, e, __fmaf_rn(__fadd_rn(s, s), e, __fmaf_rn(s, s, -p[c])));
  }
  auto two_sum = [](float x, float y, float& e) {
    const float s = __fadd_rn(x, y), t = __fsub_rn(s, x);
    e = __fadd_rn(__fsub_rn(x, __fsub_rn(s, t)), __fsub_rn(y, t));
    return s;
  };
  float e1, e2;
  const float s1 = two_sum(p[0], p[1], e1), s2 = two_sum(s1, p[2], e2);
  const float lo = __fadd_rn(__fadd_rn(e1, e2), __fadd_rn(__fadd_rn(pe[0], pe[1]), pe[2]));
  const float h = __fadd_rn(s2, lo), l = __fsub_rn(lo, __fsub_rn(h, s2));
  if (!(h >= 8.6736174e-19f && h <= 1.1529215e18f)) return false;   // 2^-60, 2^60
  const float y = rsqrtf(h);
  const float w = __fmul_rn(y, y), we = __fmaf_rn(y, y, -w);
  const float t = __fmul_rn(h, w), te = __fmaf_rn(h, w, -t);
  float e = __fsub_rn(__fsub_rn(1.0f, t), te);   // 1 - (h + l) y^2
  e = __fmaf_rn(-h, we, e);
  e = __fmaf_rn(-l, w, e);
  const float corr = __fmul_rn(y, __fmaf_rn(__fmul_rn(0.375f, e), e, __fmul_rn(0.5f, e)));
  // times 1 / (4 pi), as a pair
  const double c4 = 1.0 / (4.0 * 3.141592653589793);
  const float ch = (float)c4, cl = (float)(c4 - (double)(float)c4);
  const float v = __fmul_rn(y, ch);
  float ve = __fmaf_rn(y, ch, -v);
  ve = __fmaf_rn(corr, ch, ve);
  ve = __fmaf_rn(y, cl, ve);
  const float f = __fadd_rn(v, ve), rem = __fsub_rn(ve, __fsub_rn(f, v));
  const uint32_t u = __float_as_uint(f);
  const float half_ulp = __uint_as_float((u & 0x7F800000u) - (24u << 23));
  const float margin = __fmaf_rn(__fmul_rn(fmaxf(ah.w, bh.w), y), 1.13686838e-13f, 4.54747351e-13f);   // 2^-43, 2^-41
  *out = f;
  return __fmaf_rn(f, margin, fabsf(rem)) < half_ulp && (u & 0x7FFFFFu) != 0u;
}

__global__ void k_split_points(SrcDev src, float4* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= src.n) return;
  float h[3], l[3], m = 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double x = src.a[i + c * src.ld];
    h[c] = (float)x;
    l[c] = (float)(x - (double)h[c]);
    m = fmaxf(m, fabsf(h[c]));
  }
  out[2 * i] = make_float4(h[0], h[1], h[2], m);
  out[2 * i + 1] = make_float4(l[0], l[1], l[2], 0.f);
}

// double -> float, round to nearest even, on the integer pipe (the conversion
// instruction runs at the FP64 pipe's rate); ok is cleared where the value is
// not a normal float before the rounding
__device__ __forceinline__ float f32_of(double x, bool& ok) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t ax = hi & 0x7FFFFFFFu;
  ok = ok && ax - 0x38100000u < 0x0FD00000u;   // 2^-126 .. 2^127: no overflow by the carry
  const uint32_t t = __funnelshift_l(lo, hi, 3) - 0xC0000000u;
  const uint32_t up = (lo << 3) + (t & 1u) > 0x80000000u ? 1u : 0u;
  return __uint_as_float(((t + up) & 0x7FFFFFFFu) | (hi & 0x80000000u));
}

// The EV entries (row, k .. k + EV - 1) of A - D^(L) (trans: of its transpose)
// as the chunks of their terms; lo, hi: the row's leaf.
template <int PREC, bool TRANS>
__device__ __forceinline__ void entry_chunk(const SrcDev& src, int gr, int k, int lo, int hi, uint4* chunk) {
  using SP = Split<PREC>;
  constexpr int EV = SP::EV;
  const int n = src.n;
  if (src.pts) {   // (symmetric: one evaluation for both orientations)
    float v[EV];
    const int ga = min(gr, n - 1);
    const float4 ah = src.pts[2 * ga], al = src.pts[2 * ga + 1];
    bool redo = false;
#pragma unroll
    for (int x = 0; x < EV; ++x) {
      const int gk = k + x, gp = min(gk, n - 1);
      const bool in = gr < n && gk < n && (gk < lo || gk >= hi);
      float f;
      const bool ok = laplace_f32(ah, al, src.pts[2 * gp], src.pts[2 * gp + 1], &f);
      redo |= in && !ok;
      v[x] = in ? f : 0.f;
    }
    if (redo) {   // rare: the eight again, so that the common path has no branch
#pragma unroll 1
      for (int x = 0; x < EV; ++x) {
        const int gk = k + x;
        const float f = gr < n && gk < n && (gk < lo || gk >= hi) ? to_f32(entry_gen(src, gr, gk)) : 0.f;
#pragma unroll
        for (int y = 0; y < EV; ++y)
          if (y == x) v[y] = f;
      }
    }
    SP::split(v, chunk);
    return;
  }
  if (src.kind == HSS_SRC_DENSE) {
    // (a chunk outside of the row's leaf, which is nearly all, without masks)
    double v[EV];
    const long long step = TRANS ? 1 : src.ld;
    const double* p = src.a + (TRANS ? k + gr * src.ld : gr + k * src.ld);
    if (gr < n && k + EV <= n && (k + EV <= lo || k >= hi)) {
#pragma unroll
      for (int x = 0; x < EV; ++x) v[x] = p[x * step];
    } else {
#pragma unroll
      for (int x = 0; x < EV; ++x)
        v[x] = gr < n && k + x < n && (k + x < lo || k + x >= hi) ? p[x * step] : 0.0;
    }
    float f[EV];
    bool fine = true;
#pragma unroll
    for (int x = 0; x < EV; ++x) f[x] = f32_of(v[x], fine);
    if (!fine) {   // (volatile: not to be computed ahead of the branch)
#pragma unroll
      for (int x = 0; x < EV; ++x) asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(f[x]) : "d"(v[x]));
    }
    SP::split(f, chunk);
    return;
  }
  double v[EV];
#pragma unroll
  for (int x = 0; x < EV; ++x) {
    const int gk = k + x;
    double val = 0.0;
    if (gr < n && gk < n && (gk < lo || gk >= hi)) val = TRANS ? entry_gen(src, gk, gr) : entry_gen(src, gr, gk);
    v[x] = val;
  }
  SP::split(v, chunk);
}

// ---------------------------------------------------------------------------
// Generating kernel (entries computed by the producer warps).
// Warps 0-7: generate the A tile of each stage, drain chains, write the
// result; warp 8: TMEM allocation and (lane 0) the MMA issue.  The R tile of
// each stage comes pre-packed and is moved by warp 0 lane 0 with one bulk
// copy (expect_tx on the stage barrier, which also counts the 256
// producer arrivals).
struct TcArgs {
  SrcDev src;
  int leaf;
  int trans;
  int ncols;          // sample columns of this launch
  int N;              // columns per CTA tile (32, 64 or 128)
  int tmem_cols;      // power of two >= 4 N
  int ksplit;         // CTAs along K
  int nkt;            // k-tiles of K
  int drain;          // k-tiles per accumulation chain
  const uint8_t* Rp;  // packed R tiles (ct, kt), N x BK each
  double* S;          // row-major output, row stride lds
  long long lds;
  int atomic;         // 1: add into S (pre-zeroed); 0: store
  int* err;
  const void* toep;   // Toeplitz source: its diagonals split into the T terms
                      // (entry of A_ij at (i - j) + n - 1: TF32 x 2 both terms
                      // in one 8-byte word, BF16 x 3 term-major), or NULL
};

constexpr int GEN_WARPS = 16;
// k-tiles per accumulation chain (generated entries): TF32 x 2 carries its
// chains four k-tiles long (its samples serve tolerances >= 1e-4; measured
// error of the samples below 5e-7), BF16 x 3 two (tolerances down to 1e-6)
__host__ __device__ constexpr int drain_gen(int precision) { return precision == HSS_PREC_TF32X2 ? 4 : 2; }

// The diagonals c_t of a Toeplitz matrix (A_ij = c_{i-j}: the first column
// for i >= j, the first row for i < j), t = -(n-1) .. n-1, split into the T
// terms of the mixed form exactly as the producers split an entry: the
// Toeplitz kernel assembles its tiles from them.  TF32 x 2: the
// two terms of a diagonal side by side (one 8-byte word); BF16 x 3: term
// after term (2n - 1 entries each).
template <int PREC>
__global__ void k_toeplitz_terms(const double* col, const double* row, int n, void* out) {
  using SP = Split<PREC>;
  constexpr int T = SP::T, EV = SP::EV;
  const long long len = 2LL * n - 1;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < len; q += (long long)gridDim.x * blockDim.x) {
    const long long t = q - (n - 1);
    double v[EV];
    const double x = t >= 0 ? col[t] : row[-t];
#pragma unroll
    for (int e = 0; e < EV; ++e) v[e] = x;
    uint4 ch[T];
    SP::split(v, ch);
    if constexpr (PREC == HSS_PREC_TF32X2) {
      ((uint2*)out)[q] = make_uint2(ch[0].x, ch[1].x);
    } else {
#pragma unroll
      for (int k = 0; k < T; ++k) ((uint16_t*)out)[k * len + q] = (uint16_t)(ch[k].x & 0xFFFFu);
    }
  }
}
constexpr int GEN_THREADS = GEN_WARPS * 32 + 32;

template <int PREC, int NH, int TRANS>
__global__ void __maxnreg__(96) k_sample_tc_gen(TcArgs a) {
  using SP = Split<PREC>;
  constexpr int T = SP::T, EV = SP::EV, BK = SP::BK, KC = BK / EV;
  constexpr int DR = drain_gen(PREC);
  constexpr int NP = GEN_WARPS * 32;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int n = a.src.n, N = a.N;
  const uint32_t tileB = (uint32_t)N * 128u;
  const uint32_t stage_bytes = T * TILE_A_BYTES + tileB;
  uint64_t* full = (uint64_t*)(smem + NSTAGE * stage_bytes);
  uint64_t* empty = full + NSTAGE;
  uint64_t* tfull = empty + NSTAGE;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = (uint32_t*)(tempty + 2);
  int* lrow_lo = (int*)(tmem_slot + 4);
  int* lrow_hi = lrow_lo + BM;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int rb = blockIdx.x, ct = blockIdx.y;
  const int row0 = rb * BM, col0 = ct * N;
  const int kt0 = (int)((long long)a.nkt * blockIdx.z / a.ksplit);
  const int kt1 = (int)((long long)a.nkt * (blockIdx.z + 1) / a.ksplit);
  const int nk = kt1 - kt0;
  const int nchain = (nk + DR - 1) / DR;
  if (tid == 0) {
    for (int s = 0; s < NSTAGE; ++s) { mbar_init(&full[s], NP + 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], GEN_WARPS); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < BM) {
    int r = row0 + tid, lo = 0x7fffffff, hi = 0x7fffffff;
    if (r < n) leaf_range(r, n, a.leaf, lo, hi);
    lrow_lo[tid] = lo;
    lrow_hi[tid] = hi;
  }
  if (warp == GEN_WARPS) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"((uint32_t)a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint8_t* gB = a.Rp + ((size_t)ct * a.nkt + kt0) * tileB;

  if (warp < GEN_WARPS) {
    const int q = warp % 4, h = warp / 4;
    float s[NH], e[NH];
#pragma unroll
    for (int j = 0; j < NH; ++j) { s[j] = 0.f; e[j] = 0.f; }
    bool ok = true;
    int drained = 0;   // chains drained so far
    int st = 0;
    uint32_t ph = 0u;
    for (int it = 0; it < nk && ok; ++it) {
      if (it > 0 && ++st == NSTAGE) { st = 0; ph ^= 1u; }
      if (!mbar_wait_warp(&empty[st], ph ^ 1u, a.err, 2)) { ok = false; break; }
      uint8_t* sp = smem + st * stage_bytes;
      if (tid == 0) {
        mbar_expect_tx(&full[st], tileB);
        bulk_g2s(sp + T * TILE_A_BYTES, gB + (size_t)it * tileB, tileB, &full[st]);
      }
      const int k0 = (kt0 + it) * BK;
      for (int u = tid; u < BM * KC; u += NP) {
        int r, c;
        if (!TRANS) { r = u % BM; c = u / BM; }
        else { r = (u / (8 * KC)) * 8 + (u % 8); c = (u / 8) % KC; }
        uint4 chunk[T];
        entry_chunk<PREC, TRANS != 0>(a.src, row0 + r, k0 + c * EV, lrow_lo[r], lrow_hi[r], chunk);
        const uint32_t off = (uint32_t)(r / 8) * 1024u + (uint32_t)c * 128u + (uint32_t)(r % 8) * 16u;
#pragma unroll
        for (int t = 0; t < T; ++t) *(uint4*)(sp + t * TILE_A_BYTES + off) = chunk[t];
      }
      fence_async_smem();
      mbar_arrive(&full[st]);
      // after the last tile of chain c, drain chain c-1
      const int c = it / DR;
      if ((it % DR == DR - 1 || it == nk - 1) && c >= 1) {
        const int cd = c - 1, b = cd & 1;
        if (!mbar_wait_warp(&tfull[b], (uint32_t)(cd >> 1) & 1u, a.err, 6)) { ok = false; break; }
        tc_fence_after();
        drain_chain<NH>(tmem, N, b, q, h, s, e);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[b]);
        drained = c;
      }
    }
    // drain what is left (the last chain)
    for (int cd = drained; ok && cd < nchain; ++cd) {
      const int b = cd & 1;
      if (!mbar_wait_warp(&tfull[b], (uint32_t)(cd >> 1) & 1u, a.err, 7)) { ok = false; break; }
      tc_fence_after();
      drain_chain<NH>(tmem, N, b, q, h, s, e);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[b]);
    }
    if (ok) store_row<NH>(a.S, a.lds, n, a.ncols, row0 + 32 * q + lane, col0 + h * NH, a.atomic, s, e);
  } else if (lane == 0) {
    // ------------------------------------------------------------- MMA issuer
    const uint32_t id = idesc(SP::FMT, (uint32_t)N);
    int st = 0;
    uint32_t ph = 0u;
    for (int it = 0; it < nk; ++it) {
      if (it > 0 && ++st == NSTAGE) { st = 0; ph ^= 1u; }
      const int c = it / DR, b = c & 1;
      const bool first = (it % DR) == 0;
      if (first && !mbar_wait(&tempty[b], ((uint32_t)(c >> 1) & 1u) ^ 1u, a.err, 8)) break;
      if (!mbar_wait(&full[st], ph, a.err, 3)) break;
      tc_fence_after();
      mma_ktile<PREC>(smem_u32(smem + st * stage_bytes), tmem, N, b, first, id);
      mma_commit(&empty[st]);
      if (it % DR == DR - 1 || it == nk - 1) mma_commit(&tfull[b]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == GEN_WARPS) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"((uint32_t)a.tmem_cols)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// Toeplitz kernel.  A tile of a Toeplitz matrix is made of few different core
// matrices (8 rows x 16 bytes): the one of row group R and K chunk c holds the
// diagonals around 8 R - EV c (EV elements per chunk), so a 128 x BK tile has
// 15 (8 / EV) + BK / EV of them instead of 16 BK / EV, and the tile of the next
// k-tile shifts by BK / EV.  The producers therefore write one strip of core
// matrices, in the order of their diagonal, for up to J k-tiles at a time (an
// epoch), and the tensor core reads every tile out of it: stepping R by one
// moves the shared-memory address by SBO = 8 / EV core matrices, stepping c
// back by one moves it by LBO = one.  c runs backwards in the strip, so the two
// chunks of an MMA come in swapped order, in R as well (packed with the chunks
// of a pair exchanged): the sum of an MMA is the same.  What the strip cannot
// hold, k-tiles that meet the rows' leaf blocks or reach past n, is staged
// as whole masked tiles, one per epoch.
//
// Assembling every tile from a window of diagonals (sixteen warps, 2048 stores
// of 16 bytes per k-tile) bounded the sampling at 1700 clocks per k-tile and
// column tile; the strip takes about 100 stores per k-tile, which leaves the
// TF32 MMAs (8 of 128 x 128 x 8, 512 clocks), the R tile's bulk copy (16 KB)
// and the drains.  Two warps write the strips (drain warps that wrote them kept
// the tensor core waiting for its buffers: 61 -> 32 ms at n = 131072 and 256
// columns, in warps of their own 27 ms, 0.67 of the measured tensor rate).
constexpr int TP_NSB = 6;     // stages of R tiles
constexpr int TP_STRIP = 2;   // strip warps
constexpr int TP_THREADS = (GEN_WARPS + 2 + TP_STRIP) * 32;   // drains, copies, MMAs, strips

template <int PREC>
constexpr int toep_cores() { return 15 * (8 / Split<PREC>::EV) + Split<PREC>::BK / Split<PREC>::EV; }
// k-tiles per epoch: the strip of a term fits the 16 KB of a whole tile
template <int PREC>
constexpr int toep_epoch() {
  return (int)((TILE_A_BYTES / 128 - toep_cores<PREC>()) / (Split<PREC>::BK / Split<PREC>::EV)) + 1;
}

// The k-tiles [kt0, kt1) of a CTA cut into epochs.
struct ToepEpochs {
  int kt1, ku0, ku1, klast, J;   // masked: [ku0, ku1) and klast (-1: none)
  __device__ __forceinline__ int length(int kt, bool& masked) const {
    masked = (kt >= ku0 && kt < ku1) || kt == klast;
    if (masked) return 1;
    int end = kt1;
    if (kt < ku0) end = min(end, ku0);
    if (klast > kt) end = min(end, klast);
    return min(J, end - kt);
  }
};

__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(p));
  return p != 0u;
}

// TF32 x 2 with 128 columns: the columns of R are the rows of the product (the
// MMA's first operand) and the matrix tile its columns, eight of the leading
// terms and the eight of the second terms of a row group in turn, so that one
// MMA of 128 x 256 x 8 does what two of 128 x 128 x 8 did (an MMA is issued in
// about 110 clocks whatever its width; n = 131072, 256 columns: 26.8 to 22.4 ms,
// 0.84 of the measured tensor rate).  Cores of even number lie in one half of
// the buffer, the terms of each side by side, those of odd number in the other:
// a group to the next is SBO = one core matrix, a chunk to the one before LBO =
// half the buffer.
template <int PREC, int NH>
constexpr bool toep_swap() { return PREC == HSS_PREC_TF32X2 && NH == 32; }
constexpr uint32_t TP_HALF = TILE_A_BYTES;

// drain_chain for that product: lane = sample column, NH rows of the matrix
__device__ __forceinline__ void drain_swapped(uint32_t tmem, int b, int q, int h, float* s, float* e) {
  const uint32_t at = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(256 * b + 64 * h);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    float x[16];
    tmem_ld16_nw(at + 16 * c, x);
    tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < 8; ++i) ff_add(s[8 * c + i], e[8 * c + i], x[i]);
#pragma unroll
    for (int i = 0; i < 8; ++i) e[8 * c + i] = __fadd_rn(e[8 * c + i], x[8 + i]);
  }
}

template <int PREC, int NH, int TRANS>
__global__ void __maxnreg__(96) k_sample_tc_toep(TcArgs a) {
  using SP = Split<PREC>;
  constexpr int T = SP::T, EV = SP::EV, BK = SP::BK, KC = BK / EV, RS = 8 / EV;
  constexpr int DR = drain_gen(PREC);
  constexpr bool SWAP = toep_swap<PREC, NH>();
  constexpr uint32_t abuf = T * TILE_A_BYTES;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int n = a.src.n, N = a.N;
  const uint32_t tileB = (uint32_t)N * 128u;
  uint8_t* sB = smem + 2 * abuf;
  uint64_t* fullA = (uint64_t*)(sB + TP_NSB * tileB);
  uint64_t* emptyA = fullA + 2;
  uint64_t* fullB = emptyA + 2;
  uint64_t* emptyB = fullB + TP_NSB;
  uint64_t* tfull = emptyB + TP_NSB;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = (uint32_t*)(tempty + 2);
  int* lrow_lo = (int*)(tmem_slot + 4);
  int* lrow_hi = lrow_lo + BM;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int rb = blockIdx.x, ct = blockIdx.y;
  const int row0 = rb * BM, col0 = ct * N;
  const int kt0 = (int)((long long)a.nkt * blockIdx.z / a.ksplit);
  const int kt1 = (int)((long long)a.nkt * (blockIdx.z + 1) / a.ksplit);
  const int nk = kt1 - kt0;
  const int nchain = (nk + DR - 1) / DR;
  if (tid == 0) {
    for (int s = 0; s < 2; ++s) { mbar_init(&fullA[s], 32 * TP_STRIP); mbar_init(&emptyA[s], 1); }
    for (int s = 0; s < TP_NSB; ++s) { mbar_init(&fullB[s], 1); mbar_init(&emptyB[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], GEN_WARPS); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < BM) {
    int r = row0 + tid, lo = 0x7fffffff, hi = 0x7fffffff;
    if (r < n) leaf_range(r, n, a.leaf, lo, hi);
    lrow_lo[tid] = lo;
    lrow_hi[tid] = hi;
  }
  if (warp == GEN_WARPS) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"((uint32_t)a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // the leaves of the CTA's first and last row bound the masked k-tiles
  ToepEpochs ep;
  ep.kt1 = kt1;
  ep.ku0 = lrow_lo[0] / BK;
  ep.ku1 = (lrow_hi[min(BM, n - row0) - 1] + BK - 1) / BK;
  ep.klast = n % BK ? a.nkt - 1 : -1;
  ep.J = toep_epoch<PREC>();

  if (warp < GEN_WARPS) {
    const int q = warp % 4, h = warp / 4;
    float s[NH], e[NH];
#pragma unroll
    for (int j = 0; j < NH; ++j) { s[j] = 0.f; e[j] = 0.f; }
    bool ok = true;
    for (int cd = 0; cd < nchain; ++cd) {
      const int b = cd & 1;
      if (!mbar_wait_warp(&tfull[b], (uint32_t)(cd >> 1) & 1u, a.err, 6)) { ok = false; break; }
      tc_fence_after();
      if constexpr (SWAP) drain_swapped(tmem, b, q, h, s, e);
      else drain_chain<NH>(tmem, N, b, q, h, s, e);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[b]);
    }
    if constexpr (SWAP) {   // (store_col, written out: its call took 60 bytes more of spills, 4 % of the time)
      const int col = col0 + 32 * q + lane;
#pragma unroll
      for (int j = 0; j < NH; ++j) {
        const int row = row0 + h * NH + j;
        if (ok && col < a.ncols && row < n) {
          const double v = f2d_exact(s[j]) + f2d_exact(e[j]);
          double* out = a.S + (long long)row * a.lds + col;
          if (a.atomic) atomicAdd(out, v);
          else *out = v;
        }
      }
    } else if (ok) {
      store_row<NH>(a.S, a.lds, n, a.ncols, row0 + 32 * q + lane, col0 + h * NH, a.atomic, s, e);
    }
  } else if (warp >= GEN_WARPS + 2) {
    // ------------------------------------------------------------ strips of A
    const int tl = tid - (GEN_WARPS + 2) * 32;
    const uint2* tterm64 = (const uint2*)a.toep + (n - 1);
    const uint16_t* tterm16 = (const uint16_t*)a.toep + (n - 1);
    const long long tlen = 2LL * n - 1;
    // the EV elements of diagonals t, t + dt, ... as the chunks of the terms
    auto chunk_of = [&](int t, int dt, uint4* out, auto&& keep) {
      if constexpr (PREC == HSS_PREC_TF32X2) {
        uint2 w[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int tx = t + dt * x;
          w[x] = keep(x) && tx > -n && tx < n ? tterm64[tx] : make_uint2(0u, 0u);
        }
        out[0] = make_uint4(w[0].x, w[1].x, w[2].x, w[3].x);
        out[T - 1] = make_uint4(w[0].y, w[1].y, w[2].y, w[3].y);
      } else {
#pragma unroll
        for (int k = 0; k < T; ++k) {
          uint32_t w[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const int ta = t + dt * (2 * x), tb = ta + dt;
            const uint32_t lo = keep(2 * x) && ta > -n && ta < n ? tterm16[k * tlen + ta] : 0u;
            const uint32_t hi = keep(2 * x + 1) && tb > -n && tb < n ? tterm16[k * tlen + tb] : 0u;
            w[x] = lo | (hi << 16);
          }
          out[k] = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
    };
    auto produce = [&](int idx, int kt, int len, bool masked) -> bool {
      const int buf = idx & 1;
      if (!mbar_wait_warp(&emptyA[buf], ((uint32_t)(idx >> 1) & 1u) ^ 1u, a.err, 2)) return false;
      uint8_t* dst = smem + buf * abuf;
      if (!masked) {
        // core matrix m of the strip: diagonals d + rho - x, d = row0 - (last
        // k-tile's first column) + EV (m - (KC - 1))
        const int d0 = row0 - (kt + len - 1) * BK - EV * (KC - 1), cores = toep_cores<PREC>() + KC * (len - 1);
#pragma unroll 4
        for (int u = tl; u < cores * 8; u += 32 * TP_STRIP) {
          const int m = u / 8, rho = u % 8, d = d0 + EV * m + rho;
          uint4 ch[T];
          chunk_of(TRANS ? -d : d, TRANS ? 1 : -1, ch, [](int) { return true; });
#pragma unroll
          for (int t = 0; t < T; ++t) {
            const uint32_t off = SWAP ? (uint32_t)(m & 1) * TP_HALF + (uint32_t)((m & ~1) + t) * 128u + (uint32_t)rho * 16u
                                      : t * TILE_A_BYTES + (uint32_t)u * 16u;
            *(uint4*)(dst + off) = ch[t];
          }
        }
      } else {
        const int k0 = kt * BK;
        for (int u = tl; u < BM * KC; u += 32 * TP_STRIP) {
          const int r = u % BM, c = u / BM, gr = row0 + r, lo = lrow_lo[r], hi = lrow_hi[r];
          const int d = gr - k0 - c * EV;
          uint4 ch[T];
          chunk_of(TRANS ? -d : d, TRANS ? 1 : -1, ch, [&](int x) {
            const int gk = k0 + c * EV + x;
            return gr < n && gk < n && (gk < lo || gk >= hi);
          });
          // (swapped: the groups of a chunk together, 4 KB a chunk)
          const uint32_t off = SWAP ? (uint32_t)(c ^ 1) * 4096u + (uint32_t)(r / 8) * 256u + (uint32_t)(r % 8) * 16u
                                    : (uint32_t)(r / 8) * 1024u + (uint32_t)(c ^ 1) * 128u + (uint32_t)(r % 8) * 16u;
#pragma unroll
          for (int t = 0; t < T; ++t) *(uint4*)(dst + (SWAP ? t * 128u : t * TILE_A_BYTES) + off) = ch[t];
        }
      }
      fence_async_smem();
      mbar_arrive(&fullA[buf]);
      return true;
    };
    bool masked = false;
    for (int kt = kt0, idx = 0; kt < kt1; ++idx) {
      const int len = ep.length(kt, masked);
      if (!produce(idx, kt, len, masked)) break;
      kt += len;
    }
  } else if (warp == GEN_WARPS) {
    // ---------------------------------------------------------- copies of R
    if (lane == 0) {
      const uint8_t* gB = a.Rp + ((size_t)ct * a.nkt + kt0) * tileB;
      int st = 0;
      uint32_t ph = 0u;
      for (int it = 0; it < nk; ++it) {
        if (it > 0 && ++st == TP_NSB) { st = 0; ph ^= 1u; }
        if (!mbar_wait(&emptyB[st], ph ^ 1u, a.err, 4)) break;
        mbar_expect_tx(&fullB[st], tileB);
        bulk_g2s(sB + st * tileB, gB + (size_t)it * tileB, tileB, &fullB[st]);
      }
    }
  } else {
    // --------------------------------------------------------- MMA issuer
    const uint32_t id = idesc(SP::FMT, SWAP ? 256u : (uint32_t)N);
    const bool one = elect_one();
    bool ok = true, masked = false;
    int st = 0, it = 0;
    uint32_t ph = 0u;
    for (int kt = kt0, idx = 0; ok && kt < kt1; ++idx) {
      const int len = ep.length(kt, masked), buf = idx & 1;
      if (!mbar_wait_warp(&fullA[buf], (uint32_t)(idx >> 1) & 1u, a.err, 3)) break;
      const uint32_t sa = smem_u32(smem + buf * abuf);
      for (int j = 0; j < len; ++j, ++it) {
        if (it > 0 && ++st == TP_NSB) { st = 0; ph ^= 1u; }
        const int c = it / DR, b = c & 1;
        const bool first = (it % DR) == 0;
        if (first && !mbar_wait_warp(&tempty[b], ((uint32_t)(c >> 1) & 1u) ^ 1u, a.err, 8)) { ok = false; break; }
        if (!mbar_wait_warp(&fullB[st], ph, a.err, 5)) { ok = false; break; }
        tc_fence_after();
        if (one) {
          const uint64_t bd = sdesc(smem_u32(sB + st * tileB), 128u, 1024u);
          if constexpr (SWAP) {
            const uint64_t ad = masked ? sdesc(sa, 4096u, 128u)
                                       : sdesc(sa + 128u * (uint32_t)(KC - 2 + KC * (len - 1 - j)), TP_HALF, 128u);
#pragma unroll
            for (int ks = 0; ks < BK / SP::KSTEP; ++ks)
              mma<PREC>(tmem + (uint32_t)(256 * b), bd + (uint64_t)(ks * 16),
                        masked ? ad + (uint64_t)(ks * 512) : ad - (uint64_t)(ks * 16), id,
                        (first && ks == 0) ? 0u : 1u);
          } else {
            // chunk 2 ks + 1 of the tile's first row group, then LBO on to 2 ks
            const uint64_t ad = masked ? sdesc(sa, 128u, 1024u)
                                       : sdesc(sa + 128u * (uint32_t)(KC - 2 + KC * (len - 1 - j)), 128u, RS * 128u);
            const uint32_t hi = tmem + (uint32_t)((2 * b) * N), lo = hi + (uint32_t)N;
#pragma unroll
            for (int ks = 0; ks < BK / SP::KSTEP; ++ks) {
              const uint64_t ak = masked ? ad + (uint64_t)(ks * 16) : ad - (uint64_t)(ks * 16);   // 256 bytes
              const uint64_t bk = bd + (uint64_t)(ks * 16);
              mma<PREC>(hi, ak, bk, id, (first && ks == 0) ? 0u : 1u);
#pragma unroll
              for (int t = 1; t < T; ++t)
                mma<PREC>(lo, ak + (uint64_t)((t * TILE_A_BYTES) >> 4), bk, id, (first && ks == 0 && t == 1) ? 0u : 1u);
            }
          }
          mma_commit(&emptyB[st]);
          if (it % DR == DR - 1 || it == nk - 1) mma_commit(&tfull[b]);
          if (j == len - 1) mma_commit(&emptyA[buf]);
        }
        __syncwarp();
      }
      kt += len;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == GEN_WARPS) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"((uint32_t)a.tmem_cols)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// Packed path (a dense A is re-read on every pass): the operands are split
// once into canonical K-major tiles in global memory,
//   A, orientation o: tile (rb, kt) = T consecutive 16 KB term tiles at
//       ((o * nrb + rb) * nkt + kt) * T * 16 KB        (leaf diagonal zeroed)
//   R: tile (ct, kt) of N rows x BK at (ct * nkt + kt) * N * 128 bytes,
// and the main loop moves whole tiles with cp.async.bulk issued by one
// thread, completing on the stage mbarrier (expect_tx).  Warp 0 lane 0
// copies, warp 1 owns TMEM and (lane 0) issues the MMAs, warps 2-9 drain
// chains and write the result.

template <int PREC>
__global__ void __launch_bounds__(256) k_pack_a(SrcDev src, int leaf, int nrb, int nkt, uint8_t* out) {
  using SP = Split<PREC>;
  constexpr int T = SP::T, EV = SP::EV, BK = SP::BK, KC = BK / EV;
  __shared__ int rlo[BM], rhi[BM];
  const int n = src.n;
  const long long tile = blockIdx.x;
  const long long per_o = (long long)nrb * nkt;
  const int o = (int)(tile / per_o);
  const long long rem = tile % per_o;
  const int rb = (int)(rem / nkt), kt = (int)(rem % nkt);
  const int row0 = rb * BM, k0 = kt * BK;
  if (threadIdx.x < BM) {
    int r = row0 + threadIdx.x, lo = 0x7fffffff, hi = 0x7fffffff;
    if (r < n) leaf_range(r, n, leaf, lo, hi);
    rlo[threadIdx.x] = lo;
    rhi[threadIdx.x] = hi;
  }
  __syncthreads();
  uint8_t* dst = out + (size_t)tile * T * TILE_A_BYTES;
  for (int u = threadIdx.x; u < BM * KC; u += blockDim.x) {
    int r, c;
    if (!o) { r = u % BM; c = u / BM; }
    else { r = (u / (8 * KC)) * 8 + (u % 8); c = (u / 8) % KC; }
    uint4 chunk[T];
    if (o) entry_chunk<PREC, true>(src, row0 + r, k0 + c * EV, rlo[r], rhi[r], chunk);
    else entry_chunk<PREC, false>(src, row0 + r, k0 + c * EV, rlo[r], rhi[r], chunk);
    const uint32_t off = (uint32_t)(r / 8) * 1024u + (uint32_t)c * 128u + (uint32_t)(r % 8) * 16u;
#pragma unroll
    for (int t = 0; t < T; ++t) *(uint4*)(dst + t * TILE_A_BYTES + off) = chunk[t];
  }
}

// Packing by 128 x 128 blocks of A, each entry read (or evaluated), masked and
// rounded to FP32 once and then written to both tiles that hold it: the tile of
// its row, and the tile of its column, which belongs to the transposed
// orientation or, for a symmetric source (sym, blocks on and below the
// diagonal), to the same one.  k_pack_a reads a dense A once per orientation
// and evaluates every entry of a symmetric source twice.
// Bound by memory: dense, both orientations, TF32 x 2, n = 8192: 400 us by
// k_pack_a, 269 us here (0.53 GB read, 1.07 GB written: 5.9 TB/s); the Laplace
// samples of n = 12000, 128 columns, BF16 x 3: 1.00 to 0.78 ms.
template <int PREC, int KIND>
__global__ void __launch_bounds__(256, 3) k_pack_pair(SrcDev src, int leaf, int nb, int nkt, int sym, uint8_t* out) {
  using SP = Split<PREC>;
  constexpr int T = SP::T, EV = SP::EV, BK = SP::BK, KC = BK / EV, LD = BM + 4, U = 8;
  extern __shared__ float blk[];   // column j of the block at j LD: its rows contiguous, as in A
  __shared__ int ij[2];
  const int n = src.n, tid = threadIdx.x;
  if (tid == 0) {
    const unsigned t = blockIdx.x;
    int I, J;
    if (!sym) {   // neighbours in the grid read neighbouring rows of the same columns
      I = t % nb;
      J = t / nb;
    } else {      // column J holds the blocks I = J .. nb - 1
      const float b = 2.0f * nb + 1.0f;
      J = (int)((b - sqrtf(fmaxf(b * b - 8.0f * t, 0.0f))) * 0.5f);
      J = max(0, min(J, nb - 1));
      auto start = [&](int j) { return (unsigned)j * nb - (unsigned)j * (j - 1u) / 2u; };
      while (J > 0 && start(J) > t) --J;
      while (J + 1 < nb && start(J + 1) <= t) ++J;
      I = J + (int)(t - start(J));
    }
    ij[0] = I;
    ij[1] = J;
  }
  __syncthreads();
  const int I = ij[0], J = ij[1];
  {
    const int r = tid % BM, i = I * BM + r, ic = min(i, n - 1);
    int lo = 0, hi = 0x7fffffff;   // (a row past the end: all of it masked)
    if (i < n) leaf_range(i, n, leaf, lo, hi);
    const bool lap = KIND != HSS_SRC_DENSE && src.pts != nullptr;
    float4 ah = make_float4(0.f, 0.f, 0.f, 0.f), al = ah;
    if (lap) { ah = src.pts[2 * ic]; al = src.pts[2 * ic + 1]; }
#pragma unroll 1
    for (int c = tid / BM; c < BM; c += 2 * U) {
      float f[U];
      bool redo = false;
      if (KIND == HSS_SRC_DENSE) {
        double v[U];
#pragma unroll
        for (int x = 0; x < U; ++x) {
          const int j = J * BM + c + 2 * x;
          v[x] = j < n && (j < lo || j >= hi) ? src.a[ic + j * src.ld] : 0.0;
        }
        bool fine = true;
#pragma unroll
        for (int x = 0; x < U; ++x) f[x] = f32_of(v[x], fine);
        if (!fine) {   // (volatile: not to be computed ahead of the branch)
#pragma unroll
          for (int x = 0; x < U; ++x) asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(f[x]) : "d"(v[x]));
        }
      } else if (lap) {
#pragma unroll
        for (int x = 0; x < U; ++x) {
          const int j = J * BM + c + 2 * x, jc = min(j, n - 1);
          const bool in = j < n && (j < lo || j >= hi);
          float w;
          const bool ok = laplace_f32(ah, al, src.pts[2 * jc], src.pts[2 * jc + 1], &w);
          redo |= in && !ok;
          f[x] = in ? w : 0.f;
        }
      } else {
        redo = true;
      }
#pragma unroll
      for (int x = 0; x < U; ++x) blk[(c + 2 * x) * LD + r] = f[x];
      if (KIND != HSS_SRC_DENSE && redo) {
#pragma unroll 1
        for (int x = 0; x < U; ++x) {
          const int j = J * BM + c + 2 * x;
          blk[(c + 2 * x) * LD + r] = j < n && (j < lo || j >= hi) ? to_f32(entry_gen(src, ic, j)) : 0.f;
        }
      }
    }
  }
  __syncthreads();
  constexpr int NT = BM / BK;   // k-tiles of a block
  for (int u = tid; u < NT * BM * KC; u += 256) {   // rows of the block as tile rows
    const int r = u % BM, c = (u / BM) % KC, t = u / (BM * KC), kt = J * NT + t;
    if (kt >= nkt) break;
    float f[EV];
#pragma unroll
    for (int x = 0; x < EV; ++x) f[x] = blk[(t * BK + c * EV + x) * LD + r];
    uint4 chunk[T];
    SP::split(f, chunk);
    uint8_t* dst = out + ((size_t)I * nkt + kt) * (T * TILE_A_BYTES) + (r / 8) * 1024 + c * 128 + (r % 8) * 16;
#pragma unroll
    for (int p = 0; p < T; ++p) *(uint4*)(dst + p * TILE_A_BYTES) = chunk[p];
  }
  if (sym && I == J) return;
  const size_t o1 = sym ? 0 : (size_t)nb * nkt;
  for (int u = tid; u < NT * BM * KC; u += 256) {   // columns of the block as tile rows
    const int r = (u / (8 * KC)) % (BM / 8) * 8 + u % 8, c = (u / 8) % KC, t = u / (BM * KC), kt = I * NT + t;
    if (kt >= nkt) break;
    float f[EV];
#pragma unroll
    for (int x = 0; x < EV; x += 4) {
      const float4 d = *(const float4*)(blk + r * LD + t * BK + c * EV + x);
      f[x] = d.x; f[x + 1] = d.y; f[x + 2] = d.z; f[x + 3] = d.w;
    }
    uint4 chunk[T];
    SP::split(f, chunk);
    uint8_t* dst = out + (o1 + (size_t)J * nkt + kt) * (T * TILE_A_BYTES) + (r / 8) * 1024 + c * 128 + (r % 8) * 16;
#pragma unroll
    for (int p = 0; p < T; ++p) *(uint4*)(dst + p * TILE_A_BYTES) = chunk[p];
  }
}

template <int PREC>
__global__ void __launch_bounds__(256) k_pack_r(const double* R, long long ldr, int n, int ncols, int N,
                                                int nkt, int swap, uint8_t* out) {
  using SP = Split<PREC>;
  constexpr int EV = SP::EV, BK = SP::BK, KC = BK / EV;
  const int tile = blockIdx.x, ct = tile / nkt, kt = tile % nkt;
  uint8_t* dst = out + (size_t)tile * N * 128;
  for (int u = threadIdx.x; u < N * KC; u += blockDim.x) {
    const int r = (u / (8 * KC)) * 8 + (u % 8), c = (u / 8) % KC;
    const int gc = ct * N + r;
    double v[EV];
#pragma unroll
    for (int x = 0; x < EV; ++x) {
      const int gk = kt * BK + c * EV + x;
      v[x] = (gc < ncols && gk < n) ? R[(long long)gk + (long long)gc * ldr] : 0.0;
    }
    const uint32_t off = (uint32_t)(r / 8) * 1024u + (uint32_t)(c ^ swap) * 128u + (uint32_t)(r % 8) * 16u;
    *(uint4*)(dst + off) = SP::pack_r(v);
  }
}

struct TcPackedArgs {
  const uint8_t* A;
  const uint8_t* Rp;
  int n, nrb, nkt, N, ncols, tmem_cols, ksplit, trans, drain;
  double* S;
  double* Sc;         // the transposed orientation (trans = 0), or NULL: only S
  long long lds;
  int atomic;
  int* err;
};

template <int PREC>
constexpr int packed_stages() { return PREC == HSS_PREC_TF32X2 ? 4 : 3; }

constexpr int PK_THREADS = 18 * 32;   // copy warp, MMA warp, 16 drain warps

template <int PREC, int NH>
__global__ void __maxnreg__(96) k_sample_tc_packed(TcPackedArgs a) {
  using SP = Split<PREC>;
  constexpr int T = SP::T, NS = packed_stages<PREC>();
  extern __shared__ __align__(1024) uint8_t smem[];
  const int N = a.N;
  const uint32_t tileB = (uint32_t)N * 128u;
  const uint32_t stage_bytes = T * TILE_A_BYTES + tileB;
  uint64_t* full = (uint64_t*)(smem + NS * stage_bytes);
  uint64_t* empty = full + NS;
  uint64_t* tfull = empty + NS;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = (uint32_t*)(tempty + 2);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  // column tiles vary fastest across the grid: the CTAs that stream one
  // row block of A for different column tiles run together and share it
  // through L2, so A crosses HBM once per pass
  // (both orientations, where both are wanted, in one launch: one last wave
  // instead of two)
  const int side = blockIdx.y >= (unsigned)a.nrb ? 1 : 0, rb = blockIdx.y - side * a.nrb, ct = blockIdx.x;
  const int kt0 = (int)((long long)a.nkt * blockIdx.z / a.ksplit);
  const int kt1 = (int)((long long)a.nkt * (blockIdx.z + 1) / a.ksplit);
  const int nk = kt1 - kt0, DR = a.drain;
  const int nchain = (nk + DR - 1) / DR;
  if (tid == 0) {
    for (int s = 0; s < NS; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], 16); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"((uint32_t)a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint8_t* gA = a.A + ((size_t)((a.trans + side) * a.nrb + rb) * a.nkt + kt0) * (T * TILE_A_BYTES);
  const uint8_t* gB = a.Rp + ((size_t)ct * a.nkt + kt0) * tileB;
  if (warp == 0) {
    if (lane == 0) {
      for (int it = 0; it < nk; ++it) {
        const int s = it % NS;
        const uint32_t ph = (uint32_t)(it / NS) & 1u;
        if (!mbar_wait(&empty[s], ph ^ 1u, a.err, 12)) break;
        uint8_t* st = smem + s * stage_bytes;
        mbar_expect_tx(&full[s], stage_bytes);
#pragma unroll
        for (int t = 0; t < T; ++t)
          bulk_g2s(st + t * TILE_A_BYTES, gA + (size_t)it * (T * TILE_A_BYTES) + t * TILE_A_BYTES,
                   TILE_A_BYTES, &full[s]);
        bulk_g2s(st + T * TILE_A_BYTES, gB + (size_t)it * tileB, tileB, &full[s]);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t id = idesc(SP::FMT, (uint32_t)N);
      for (int it = 0; it < nk; ++it) {
        const int s = it % NS;
        const uint32_t ph = (uint32_t)(it / NS) & 1u;
        const int c = it / DR, b = c & 1;
        const bool first = (it % DR) == 0;
        if (first && !mbar_wait(&tempty[b], ((uint32_t)(c >> 1) & 1u) ^ 1u, a.err, 15)) break;
        if (!mbar_wait(&full[s], ph, a.err, 13)) break;
        tc_fence_after();
        if constexpr (NH == 32) mma_ktile_swapped<PREC>(smem_u32(smem + s * stage_bytes), tmem, b, first);   // N = 128
        else mma_ktile<PREC>(smem_u32(smem + s * stage_bytes), tmem, N, b, first, id);
        mma_commit(&empty[s]);
        if (it % DR == DR - 1 || it == nk - 1) mma_commit(&tfull[b]);
      }
    }
  } else {
    // --------------------------------------------------------- drain warps
    const int q = warp % 4, h = (warp - 2) / 4;
    float s[NH], e[NH];
#pragma unroll
    for (int j = 0; j < NH; ++j) { s[j] = 0.f; e[j] = 0.f; }
    bool ok = true;
    for (int cd = 0; cd < nchain; ++cd) {
      const int b = cd & 1;
      if (!mbar_wait_warp(&tfull[b], (uint32_t)(cd >> 1) & 1u, a.err, 14)) { ok = false; break; }
      tc_fence_after();
      drain_chain<NH>(tmem, N, b, q, h, s, e);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[b]);
    }
    if (ok && nk > 0) {
      double* S = side ? a.Sc : a.S;
      if constexpr (NH == 32) store_col<NH>(S, a.lds, a.n, a.ncols, rb * BM + h * NH, ct * N + 32 * q + lane, a.atomic, s, e);
      else store_row<NH>(S, a.lds, a.n, a.ncols, rb * BM + 32 * q + lane, ct * N + h * NH, a.atomic, s, e);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"((uint32_t)a.tmem_cols)
                 : "memory");
  }
}

int tile_n(int ncols) { return ncols <= 64 ? 64 : 128; }

int tmem_cols_for(int N) {
  int tc = 32;
  while (tc < 4 * N) tc *= 2;
  return tc;
}

constexpr int DRAIN_PACKED = 2;   // k-tiles per accumulation chain (dense, packed)

template <int PREC>
cudaError_t launch_packed_t(const TcPackedArgs& a, int gx, int gy, cudaStream_t st) {
  constexpr int T = Split<PREC>::T, NS = packed_stages<PREC>();
  const size_t sm = (size_t)NS * (T * TILE_A_BYTES + (size_t)a.N * 128) + 8 * (2 * NS + 4) + 16 + 1024;
  dim3 grid(gy, gx, a.ksplit);   // x: column tiles, y: row blocks (of both orientations)
#define HSS_LAUNCH_PK(NHV)                                                                          \
  do {                                                                                              \
    cudaError_t e = cudaFuncSetAttribute(k_sample_tc_packed<PREC, NHV>,                             \
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);     \
    if (e != cudaSuccess) return e;                                                                 \
    k_sample_tc_packed<PREC, NHV><<<grid, PK_THREADS, sm, st>>>(a);                                 \
  } while (0)
  if (a.N == 64) HSS_LAUNCH_PK(16);
  else HSS_LAUNCH_PK(32);
#undef HSS_LAUNCH_PK
  return cudaGetLastError();
}

template <int PREC>
cudaError_t launch_gen_t(const TcArgs& a, int gx, int gy, cudaStream_t st) {
  constexpr int T = Split<PREC>::T;
  const dim3 grid(gx, gy, a.ksplit);
  const bool toep = a.toep != nullptr;
  const size_t sm = toep ? (size_t)2 * T * TILE_A_BYTES + (size_t)TP_NSB * a.N * 128 + 8 * (2 * TP_NSB + 8) + 16 +
                               2 * BM * sizeof(int) + 1024
                         : (size_t)NSTAGE * (T * TILE_A_BYTES + (size_t)a.N * 128) + 8 * (2 * NSTAGE + 4) + 16 +
                               2 * BM * sizeof(int) + 1024;
  auto run = [&](auto* kernel, int threads) -> cudaError_t {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kernel<<<grid, threads, sm, st>>>(a);
    return cudaGetLastError();
  };
  if (toep) {
    if (a.N == 64)
      return a.trans ? run(k_sample_tc_toep<PREC, 16, 1>, TP_THREADS) : run(k_sample_tc_toep<PREC, 16, 0>, TP_THREADS);
    return a.trans ? run(k_sample_tc_toep<PREC, 32, 1>, TP_THREADS) : run(k_sample_tc_toep<PREC, 32, 0>, TP_THREADS);
  }
  if (a.N == 64)
    return a.trans ? run(k_sample_tc_gen<PREC, 16, 1>, GEN_THREADS) : run(k_sample_tc_gen<PREC, 16, 0>, GEN_THREADS);
  return a.trans ? run(k_sample_tc_gen<PREC, 32, 1>, GEN_THREADS) : run(k_sample_tc_gen<PREC, 32, 0>, GEN_THREADS);
}

int bk_of(int precision) { return precision == HSS_PREC_TF32X2 ? 32 : 64; }

// K split across CTAs: enough CTAs for `waves` waves, but at least 64 k-tiles
// per CTA so that the epilogue (one pass over the 128 x N tile) stays small
// against the main loop.
int ksplit_for(int gx, int gy, int nkt, int waves) {
  int ks = (waves * 152 + gx * gy - 1) / (gx * gy);
  const int cap = nkt / 64;
  if (ks > cap) ks = cap;
  return ks < 1 ? 1 : ks;
}

}  // namespace

cudaError_t launch_split_points(const SrcDev& src, float4* out, cudaStream_t st) {
  if (src.kind != HSS_SRC_LAPLACE || src.n <= 0) return cudaErrorInvalidValue;
  k_split_points<<<(src.n + 127) / 128, 128, 0, st>>>(src, out);
  return cudaGetLastError();
}

size_t toeplitz_terms_bytes(int n, int precision) {
  return (size_t)(2LL * n - 1) * (precision == HSS_PREC_TF32X2 ? 2 * 4 : 3 * 2);
}

cudaError_t launch_toeplitz_terms(const SrcDev& src, int precision, void* out, cudaStream_t st) {
  if (src.kind != HSS_SRC_TOEPLITZ || src.n <= 0) return cudaErrorInvalidValue;
  const long long len = 2LL * src.n - 1;
  const unsigned grid = (unsigned)std::min<long long>((len + 255) / 256, 152LL * 16);
  if (precision == HSS_PREC_TF32X2) k_toeplitz_terms<HSS_PREC_TF32X2><<<grid, 256, 0, st>>>(src.a, src.b, src.n, out);
  else if (precision == HSS_PREC_BF16X3) k_toeplitz_terms<HSS_PREC_BF16X3><<<grid, 256, 0, st>>>(src.a, src.b, src.n, out);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

size_t packed_a_bytes(int n, int precision, int orients) {
  const int T = precision == HSS_PREC_TF32X2 ? 2 : 3, bk = bk_of(precision);
  const size_t nrb = (n + BM - 1) / BM, nkt = (n + bk - 1) / bk;
  return orients * nrb * nkt * T * (size_t)TILE_A_BYTES;
}

size_t packed_r_bytes(int n, int ncols, int precision) {
  const int bk = bk_of(precision);
  const int N = tile_n(ncols);
  const size_t nct = (ncols + N - 1) / N, nkt = (n + bk - 1) / bk;
  return nct * nkt * (size_t)N * 128;
}

cudaError_t launch_pack_a(const SrcDev& src, int leaf, int precision, int orients, void* out, cudaStream_t st) {
  if (src.kind < HSS_SRC_DENSE || src.kind > HSS_SRC_LAPLACE) return cudaErrorInvalidValue;   // no entries on the device
  const int n = src.n;
  const int bk = bk_of(precision);
  const int nrb = (n + BM - 1) / BM, nkt = (n + bk - 1) / bk;
  const long long tiles = (long long)orients * nrb * nkt;
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  // by blocks where a block serves two tiles; a dense A wanted in one
  // orientation is read once either way (and may be symmetric only in name)
  const bool dense = src.kind == HSS_SRC_DENSE, sym = src.kind == HSS_SRC_GAUSS || src.kind == HSS_SRC_LAPLACE;
  if ((dense && orients == 2) || (sym && orients == 1)) {
    auto run = [&](auto* kernel) -> cudaError_t {
      const int sm = BM * (BM + 4) * (int)sizeof(float);
      const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
      if (e != cudaSuccess) return e;
      const long long grid = dense ? (long long)nrb * nrb : (long long)nrb * (nrb + 1) / 2;
      kernel<<<(unsigned)grid, 256, sm, st>>>(src, leaf, nrb, nkt, dense ? 0 : 1, (uint8_t*)out);
      return cudaGetLastError();
    };
    if (precision == HSS_PREC_TF32X2)
      return dense ? run(k_pack_pair<HSS_PREC_TF32X2, HSS_SRC_DENSE>) : run(k_pack_pair<HSS_PREC_TF32X2, HSS_SRC_LAPLACE>);
    return dense ? run(k_pack_pair<HSS_PREC_BF16X3, HSS_SRC_DENSE>) : run(k_pack_pair<HSS_PREC_BF16X3, HSS_SRC_LAPLACE>);
  }
  if (precision == HSS_PREC_TF32X2)
    k_pack_a<HSS_PREC_TF32X2><<<(unsigned)tiles, 256, 0, st>>>(src, leaf, nrb, nkt, (uint8_t*)out);
  else
    k_pack_a<HSS_PREC_BF16X3><<<(unsigned)tiles, 256, 0, st>>>(src, leaf, nrb, nkt, (uint8_t*)out);
  return cudaGetLastError();
}

cudaError_t launch_pack_r(const double* R, long long ldr, int n, int ncols, int precision, bool toep,
                          void* out, cudaStream_t st) {
  if (n <= 0 || ncols <= 0) return cudaSuccess;
  const int bk = bk_of(precision), swap = toep ? 1 : 0;
  const int N = tile_n(ncols), nct = (ncols + N - 1) / N, nkt = (n + bk - 1) / bk;
  if (precision == HSS_PREC_TF32X2)
    k_pack_r<HSS_PREC_TF32X2><<<nct * nkt, 256, 0, st>>>(R, ldr, n, ncols, N, nkt, swap, (uint8_t*)out);
  else
    k_pack_r<HSS_PREC_BF16X3><<<nct * nkt, 256, 0, st>>>(R, ldr, n, ncols, N, nkt, swap, (uint8_t*)out);
  return cudaGetLastError();
}

int sample_tc_packed_ksplit(int n, int ncols, int precision) {
  const int N = tile_n(ncols);
  const int gx = (n + BM - 1) / BM, gy = (ncols + N - 1) / N, nkt = (n + bk_of(precision) - 1) / bk_of(precision);
  return ksplit_for(gx, gy, nkt, tuning_get().sample_waves_packed);
}

int sample_tc_ksplit(int n, int ncols, int precision) {
  const int N = tile_n(ncols);
  const int gx = (n + BM - 1) / BM, gy = (ncols + N - 1) / N, nkt = (n + bk_of(precision) - 1) / bk_of(precision);
  return ksplit_for(gx, gy, nkt, tuning_get().sample_waves_generated);
}

cudaError_t launch_sample_tc_packed(const void* A, const void* Rp, int n, int ncols, int precision,
                                    int trans, int ksplit, double* S, double* Sc, long long lds, int* err,
                                    cudaStream_t st) {
  if (n <= 0 || ncols <= 0) return cudaSuccess;
  TcPackedArgs a;
  a.A = (const uint8_t*)A;
  a.Rp = (const uint8_t*)Rp;
  a.n = n;
  a.nrb = (n + BM - 1) / BM;
  a.nkt = (n + bk_of(precision) - 1) / bk_of(precision);
  a.N = tile_n(ncols);
  a.ncols = ncols;
  a.tmem_cols = tmem_cols_for(a.N);
  a.ksplit = ksplit;
  a.trans = trans;
  a.drain = DRAIN_PACKED;
  a.S = S;
  a.Sc = Sc;
  a.lds = lds;
  a.atomic = a.ksplit > 1 ? 1 : 0;
  a.err = err;
  const int gy = (ncols + a.N - 1) / a.N, gx = (Sc ? 2 : 1) * a.nrb;
  if (precision == HSS_PREC_TF32X2) return launch_packed_t<HSS_PREC_TF32X2>(a, gx, gy, st);
  if (precision == HSS_PREC_BF16X3) return launch_packed_t<HSS_PREC_BF16X3>(a, gx, gy, st);
  return cudaErrorInvalidValue;
}

// S (+)= (A - D^(L))^{[T]} R with entries generated by the producer warps;
// Rp holds R packed by launch_pack_r; S must be zeroed by the caller when the
// K range is split across CTAs (*used_atomic).
cudaError_t launch_sample_tc(const SrcDev& src, int leaf, int precision, int trans, int ncols,
                             const void* Rp, double* S, long long lds, int* err, int* used_atomic,
                             const void* toep, cudaStream_t st) {
  if (src.kind < HSS_SRC_DENSE || src.kind > HSS_SRC_LAPLACE) return cudaErrorInvalidValue;   // no entries on the device
  const int n = src.n;
  if (n <= 0 || ncols <= 0) return cudaSuccess;
  TcArgs a;
  a.src = src;
  a.leaf = leaf;
  a.trans = trans;
  a.ncols = ncols;
  a.N = tile_n(ncols);
  a.tmem_cols = tmem_cols_for(a.N);
  a.nkt = (n + bk_of(precision) - 1) / bk_of(precision);
  const int gx = (n + BM - 1) / BM, gy = (ncols + a.N - 1) / a.N;
  a.ksplit = sample_tc_ksplit(n, ncols, precision);
  a.drain = drain_gen(precision);
  a.Rp = (const uint8_t*)Rp;
  a.S = S;
  a.lds = lds;
  a.atomic = a.ksplit > 1 ? 1 : 0;
  a.err = err;
  a.toep = src.kind == HSS_SRC_TOEPLITZ ? toep : nullptr;
  *used_atomic = a.atomic;
  if (precision == HSS_PREC_TF32X2) return launch_gen_t<HSS_PREC_TF32X2>(a, gx, gy, st);
  if (precision == HSS_PREC_BF16X3) return launch_gen_t<HSS_PREC_BF16X3>(a, gx, gy, st);
  return cudaErrorInvalidValue;
}

}  // namespace hss
