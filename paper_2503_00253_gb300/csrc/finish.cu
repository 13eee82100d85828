// a9-a11: quadrature-weighted accumulation and the state-space update.
//
//   vbar^(i) = R^-1/2 sum_q p_q u_q^(i)                       (Sec. 3.2, App. E)
//   z_a^(i)  = z^(i) - Sxh vbar^(i),  A_a = sqrt(N-1) Z_a       (Sec. 3.2)
//   mu_a     = mu + Sxh R^-1/2 u_mean                           (Eq. info_esrf_mean_solve)
//
// The quadrature sum is FP64.  Sxh is the state-obs band formed in setup, so
// the state update is one banded product with N + 1 right-hand sides.
#include "common.cuh"
#include "internal.h"

namespace infoesrf {

// 32 observations x kAccCols columns per CTA: a warp per column with its lanes
// over observations (coalesced rows of U), written back through shared memory so
// that Vbar's rows get whole sectors.  (With the columns fastest every read
// of U touched one sector per lane.)
constexpr int kAccCols = 8;
template <typename T>
__global__ void __launch_bounds__(32 * kAccCols) k_accumulate(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.z];
  const int64_t N1 = pr.N + 1, d = pr.d;
  const int64_t a0 = (int64_t)blockIdx.x * 32, m0 = (int64_t)blockIdx.y * kAccCols;
  if (a0 >= d || m0 >= N1) return;
  __shared__ double tile[kAccCols][33];
  {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t a = a0 + lane, m = m0 + warp;
    const T* U = reinterpret_cast<const T*>(pr.U);
    double acc = 0.0;
    if (a < d && m < pr.N) {
      if (pr.do_pert) {
        const T* u = U + (pr.mean_sys + m) * d + a;
#pragma unroll 8
        for (int q = 0; q < pr.Q; ++q) acc += pr.p[q] * (double)u[(int64_t)q * pr.N * d];
      }
    } else if (a < d && m == pr.N && pr.do_mean) {
      acc = (double)U[a];   // sid 0
    }
    tile[warp][lane] = acc;
  }
  __syncthreads();
  const int64_t a = a0 + threadIdx.x / kAccCols, m = m0 + threadIdx.x % kAccCols;
  if (a >= d || m >= N1) return;
  const double v = pr.rinv[a] * tile[threadIdx.x % kAccCols][threadIdx.x / kAccCols];
  pr.Vbar[a * N1 + m] = v;
  reinterpret_cast<T*>(pr.VbarT)[a * N1 + m] = to_t<T>(v);
}

// A CTA takes 32 consecutive state points and kStateCols columns (member m < N,
// or the mean m == N); its warps take the band's entries in turn, lanes over
// points (coalesced band loads; neighbouring points share most rows of Vbar),
// and the warps' sums are added in order.  One band entry serves eight columns,
// and the chain of dependent loads of a point is a quarter of its entries.
// (One thread per point and pair of columns read the band 21 times at N = 40:
// bound by those reads and their latency.)
constexpr int kStateCols = 8, kStateWarps = 4;
template <typename T>
__global__ void __launch_bounds__(32 * kStateWarps) k_state_apply(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.z];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t x0 = (int64_t)blockIdx.x * 32, x = x0 + lane;
  const int64_t n = pr.n, N = pr.N, N1 = N + 1;
  const int64_t m0 = (int64_t)blockIdx.y * kStateCols;
  if (x0 >= n || m0 > N) return;
  const T* __restrict__ val = reinterpret_cast<const T*>(pr.xo_val);
  const int32_t* __restrict__ col = pr.xo_col;
  const T* __restrict__ Vb = reinterpret_cast<const T*>(pr.VbarT);
  const int nnz = x < n ? pr.xo_nnz[x] : 0;
  const int nc = (int)(N1 - m0 < kStateCols ? N1 - m0 : kStateCols);
  T acc[kStateCols];
#pragma unroll
  for (int j = 0; j < kStateCols; ++j) acc[j] = T(0);
#pragma unroll 4
  for (int e = warp; e < nnz; e += kStateWarps) {
    const T v = val[(int64_t)e * n + x];
    const T* vb = Vb + (int64_t)col[(int64_t)e * n + x] * N1 + m0;
#pragma unroll
    for (int j = 0; j < kStateCols; ++j)
      if (j < nc) acc[j] += v * vb[j];
  }
  __shared__ T part[kStateWarps][kStateCols][32];
#pragma unroll
  for (int j = 0; j < kStateCols; ++j) part[warp][j][lane] = acc[j];
  __syncthreads();
  if (x >= n) return;
  const double mu = pr.mu[x];
#pragma unroll
  for (int i = 0; i < kStateCols / kStateWarps; ++i) {
    const int j = warp + i * kStateWarps;
    if (j >= nc) break;
    const int64_t m = m0 + j;
    T t = part[0][j][lane];
#pragma unroll
    for (int w = 1; w < kStateWarps; ++w) t += part[w][j][lane];
    const double inc = (double)t;
    if (m < N) {
      if (pr.do_pert) pr.A_a[m * n + x] = (pr.X[m * n + x] - mu) - pr.sqrt_nm1 * inc;
    } else if (pr.do_mean) {
      pr.mu_a[x] = mu + inc;
    }
  }
}

void launch_finish(const ProblemTable& tab, const ProblemDev* dtab, cudaStream_t st, bool accumulate) {
  int64_t dmax = 0, nmax = 0, Nmax = 0;
  for (int i = 0; i < tab.count; ++i) {
    const ProblemDev& p = tab.p[i];
    dmax = p.d > dmax ? p.d : dmax;
    nmax = p.n > nmax ? p.n : nmax;
    Nmax = p.N > Nmax ? p.N : Nmax;
  }
  const dim3 ga((unsigned)((dmax + 31) / 32), (unsigned)((Nmax + kAccCols) / kAccCols), tab.count);
  const dim3 gs((unsigned)((nmax + 31) / 32), (unsigned)((Nmax + kStateCols) / kStateCols), tab.count);
  if (tab.p[0].precision == 0) {
    if (accumulate) { k_accumulate<double><<<ga, 32 * kAccCols, 0, st>>>(dtab); note_launches(1); }
    k_state_apply<double><<<gs, 32 * kStateWarps, 0, st>>>(dtab); note_launches(1);
  } else {
    if (accumulate) { k_accumulate<float><<<ga, 32 * kAccCols, 0, st>>>(dtab); note_launches(1); }
    k_state_apply<float><<<gs, 32 * kStateWarps, 0, st>>>(dtab); note_launches(1);
  }
}

}  // namespace infoesrf
