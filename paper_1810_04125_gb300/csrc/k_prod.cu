// The HSS product H X or H^T X for a moderate number of columns (section 2.1:
// up-sweep x^_tau = V_tau^T [...], coupling through B12 / B21, down-sweep with
// U_tau, leaves D_tau), one launch per tree level and direction from task
// lists that are laid out once per handle.
//
// What bounds it: for a few columns the chain of levels (a launch is 2 to 3
// us, and every level waits for the last), for more the FP64 pipe (one FMA per
// generator element and column).  The batched tile kernel spent 64 x 64 FP64
// tiles on these products whatever the number of columns (1.07 us per unit of
// K), and uploaded a job list per launch.
//
// A task is one node's result, a CTA 16 rows of it,
//   up    x^(i)   = x(piv_i) + sum_l X(i, l) x(piv_(k+l))
//   down  y^_c(i) = sum_l B(i, l) x^_sibling(l) + [U_p y^_p](row of c's i)
//   leaf  Y(i)    = sum_j D(i, j) X(j) + [U y^](i)
// with U = Pi [I; X^T] read by rows through the inverse pivot order, so that the
// coupling and the down-sweep of a node are one sum and no result is written
// twice.  A CTA takes up to RC columns.  Where the block is
// contiguous along its rows, half a warp holds the 16 rows and the sixteen
// halves split l; where it is contiguous along l (transposed blocks, rows of
// X^T), it is turned in shared memory first: with lanes along l the additions
// that join a row's lanes took as many FP64 instructions as the sums.  Partial
// sums meet in shared memory.
#include "hss_internal.h"

namespace hss {
namespace {

constexpr int PT = 256, PW = PT / 32;
constexpr int LB = 64;   // l per staged piece of a block that is contiguous along l

// x(l) of a sum: element l of the vector(s) behind it, columns at stride cs
struct Vec {
  const double* p0;   // elements below split (element stride es)
  const double* p1;
  long long es, cs;
  int split;
};
__device__ __forceinline__ const double* at(const Vec& v, int l) {
  return l < v.split ? v.p0 + (long long)l * v.es : v.p1 + (long long)(l - v.split) * v.es;
}

// Every launch of a product but the first may begin before the one before it
// has finished (programmatic dependent launch): what does not depend on it is
// read first, the node vectors after this wait.
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <int RC>
__global__ void __launch_bounds__(PT) k_prod(const ProdTask* __restrict__ tasks, int nrhs, const double* __restrict__ X,
                                             long long ldx, double* __restrict__ Y, long long ldy, double* buf) {
  __shared__ double part[PW][16][RC];
  __shared__ double tile[16][LB + 1];
  __shared__ int s_pos[16];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  ProdTask t = tasks[blockIdx.y];
  const int i0 = 16 * blockIdx.x, c0 = blockIdx.z * RC, nc = min(RC, nrhs - c0);
  if (i0 >= t.rows) return;
  t.rows = min(16, t.rows - i0);
  t.M += t.trans ? (long long)i0 * t.ld : i0;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int r = lane & 15, l00 = 2 * warp + (lane >> 4);   // row and first l of a half-warp
  if (t.k2 > 0 && tid < 16) s_pos[tid] = tid < t.rows ? t.pos[i0 + tid] : 0;
  Vec v;   // the vector of the first sum
  if (t.in_lo >= 0) {
    v.p0 = v.p1 = X + t.in_lo + (long long)c0 * ldx;
    v.es = 1;
    v.cs = ldx;
    v.split = 0x7fffffff;
  } else {
    v.p0 = buf + (long long)t.in0 * nrhs + c0;
    v.p1 = buf + (long long)t.in1 * nrhs + c0;
    v.es = nrhs;
    v.cs = 1;
    v.split = t.split;
  }
  double acc[RC];
#pragma unroll
  for (int c = 0; c < RC; ++c) acc[c] = 0.0;
  auto add = [&](double m, const double* x, long long cs) {
#pragma unroll
    for (int c = 0; c < RC; ++c)
      if (RC == 1 || c < nc) acc[c] = __fma_rn(m, x[(long long)c * cs], acc[c]);
  };
  // A block that is contiguous along l goes through shared memory in pieces of
  // LB, the next piece's loads in flight during the sums of this one; rows
  // without a pointer (skeleton rows of U) take no part.
  auto staged = [&](auto&& row_ptr, int K, const Vec& x, bool dep) {
    constexpr int NP = 16 * LB / PT;
    double nx[NP];
    auto fetch = [&](int l0) {
#pragma unroll
      for (int q = 0; q < NP; ++q) {
        const int e = tid + q * PT, row = e / LB, l = l0 + e % LB;
        const double* p = row < t.rows && l < K ? row_ptr(row) : nullptr;
        nx[q] = p ? p[l] : 0.0;
      }
    };
    fetch(0);
    if (dep) wait_previous();
    for (int l0 = 0; l0 < K; l0 += LB) {
#pragma unroll
      for (int q = 0; q < NP; ++q) tile[(tid + q * PT) / LB][(tid + q * PT) % LB] = nx[q];
      __syncthreads();
      if (l0 + LB < K) fetch(l0 + LB);
      if (r < t.rows && row_ptr(r)) {
        const int le = min(LB, K - l0);
        for (int l = l00; l < le; l += 2 * PW) add(tile[r][l], at(x, l0 + l), x.cs);
      }
      __syncthreads();
    }
  };
  // first sum
  if (t.trans) {
    staged([&](int row) { return t.M + (long long)row * t.ld; }, t.K, v, true);
  } else {
    const double* m = t.M + r;
    constexpr int UN = 4;   // loads in flight
    double a[UN];
    int g[UN];
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const int l = l00 + u * 2 * PW;
      a[u] = r < t.rows && l < t.K ? m[(long long)l * t.ld] : 0.0;
      g[u] = t.gather && l < t.K ? t.gather[l] : l;
    }
    wait_previous();
    if (r < t.rows) {
      for (int l0 = l00; l0 < t.K; l0 += UN * 2 * PW) {
        if (l0 > l00) {
#pragma unroll
          for (int u = 0; u < UN; ++u) {
            const int l = l0 + u * 2 * PW;
            a[u] = l < t.K ? m[(long long)l * t.ld] : 0.0;
            g[u] = t.gather && l < t.K ? t.gather[l] : l;
          }
        }
#pragma unroll
        for (int u = 0; u < UN; ++u)
          if (l0 + u * 2 * PW < t.K) add(a[u], at(v, g[u]), v.cs);
      }
    }
  }
  // second sum: the rows of X2^T
  if (t.k2 > 0) {
    __syncthreads();   // s_pos
    Vec y;
    y.p0 = y.p1 = buf + (long long)t.y2 * nrhs + c0;
    y.es = nrhs;
    y.cs = 1;
    y.split = 0x7fffffff;
    staged([&](int row) -> const double* {
      return s_pos[row] >= t.k2 ? t.X2 + (long long)(s_pos[row] - t.k2) * t.k2 : nullptr;
    }, t.k2, y, false);
  }
#pragma unroll
  for (int c = 0; c < RC; ++c) {
    const double s = acc[c] + __shfl_xor_sync(0xffffffffu, acc[c], 16);
    if (lane < 16) part[warp][r][c] = s;
  }
  __syncthreads();
  for (int e = tid; e < 16 * RC; e += PT) {
    const int row = e / RC, c = e % RC;
    if (row >= t.rows || c >= nc) continue;
    double s = (part[0][row][c] + part[1][row][c]) + (part[2][row][c] + part[3][row][c]);
    s += (part[4][row][c] + part[5][row][c]) + (part[6][row][c] + part[7][row][c]);
    if (t.k2 > 0 && s_pos[row] < t.k2) s += buf[(long long)(t.y2 + s_pos[row]) * nrhs + c0 + c];
    if (t.self) s += at(v, t.self[i0 + row])[(long long)c * v.cs];
    if (t.out_lo >= 0) Y[t.out_lo + i0 + row + (long long)(c0 + c) * ldy] = s;
    else buf[(long long)(t.out + i0 + row) * nrhs + c0 + c] = s;
  }
}

template <int RC>
cudaError_t launch_rc(const ProdTask* tasks, dim3 grid, bool after, int nrhs, const double* X, long long ldx, double* Y,
                      long long ldy, double* buf, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(PT);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = after ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_prod<RC>, tasks, nrhs, X, ldx, Y, ldy, buf);
}

}  // namespace

// after: the launch before this one on the stream belongs to the same product
cudaError_t launch_prod(const ProdTask* tasks, int ntasks, int tiles, bool after, int nrhs, const double* X, long long ldx,
                        double* Y, long long ldy, double* buf, cudaStream_t st) {
  if (ntasks <= 0 || tiles <= 0 || nrhs <= 0) return cudaSuccess;
  const int rc = nrhs >= 5 ? 8 : (nrhs >= 3 ? 4 : nrhs);
  for (int t0 = 0; t0 < ntasks; t0 += 65535) {   // grid y holds 65535 blocks
    const dim3 grid(tiles, ntasks - t0 < 65535 ? ntasks - t0 : 65535, (nrhs + rc - 1) / rc);
    auto* f = rc == 8 ? launch_rc<8> : rc == 4 ? launch_rc<4> : rc == 2 ? launch_rc<2> : launch_rc<1>;
    const cudaError_t e = f(tasks + t0, grid, after && t0 == 0, nrhs, X, ldx, Y, ldy, buf, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace hss
