// Setup stages of one InFo-ESRF analysis, batched over problems (blockIdx.y).
//
//  * anomalies and observation gather   (Eq. normalized_perturbations, W = H Z)
//  * localized obs covariance band C    (Eq. localized_state_covar, Sec. 2.3,
//    normalized by R^-1/2 as in App. E) and the state-obs band Sxh
//  * quadrature nodes and weights       (App. D)
//  * randomized Ritz pairs of C         (App. E, Halko et al. Alg. 5.3)
//
// Precision: T is the bulk type (double on the FP64 path, float on the mixed
// path).  Sums that feed scalars use DotAcc<T> (float-float for float).
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace infoesrf {

template <typename T>
__device__ __forceinline__ T* tp(void* p) { return reinterpret_cast<T*>(p); }
template <typename T>
__device__ __forceinline__ const T* tp(const void* p) { return reinterpret_cast<const T*>(p); }

// ---------------------------------------------------------------------------
// Problem table upload: chunks of the host table travel as kernel parameters,
// so the upload is stream-ordered and graph-capturable.
// ---------------------------------------------------------------------------
constexpr int kChunk = 4;
struct TableChunk {
  int32_t first, count;
  ProblemDev p[kChunk];
};

// One launch per chunk of problems: block (0, i) writes problem i's table entry
// and clears its scalars and status; every block fills part of its per-axis
// table of (axis distance / half-width)^2 for every index offset, which the
// band kernels use instead of a transcendental per candidate pair.  Only the
// parameter copy of the table is read, so no block waits for the upload.
// Small CTAs: the distances' FP64 sines spread over all SMs, and the entry is copied
// by words (256 threads and a copy by one thread: 4 to 6 us more a call at 240 to
// 8192 points).
constexpr int kPrepThreads = 64;
__global__ void __launch_bounds__(kPrepThreads) k_prepare(const __grid_constant__ TableChunk c, ProblemDev* dst) {
  const int i = blockIdx.y;
  if (i >= c.count) return;
  const ProblemDev& pc = c.p[i];
  static_assert(sizeof(ProblemDev) % 8 == 0, "copied by words");
  if (blockIdx.x == 0)
    for (int w = threadIdx.x; w < (int)(sizeof(ProblemDev) / 8); w += kPrepThreads)
      reinterpret_cast<uint64_t*>(dst + c.first + i)[w] = reinterpret_cast<const uint64_t*>(&pc)[w];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    pc.scal[0] = 0.0;
    pc.scal[1] = __longlong_as_double(0x7ff0000000000000LL);  // +inf, atomically lowered
    for (int u = 2; u < 8; ++u) pc.scal[u] = 0.0;
    for (int u = 0; u < 4; ++u) pc.status[u] = 0;
  }
  const GridDev& g = pc.grid;
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t total = g.ext[0] + g.ext[1] + g.ext[2];
  if (e >= total) return;
  const int ax = e < g.ext[0] ? 0 : (e < g.ext[0] + g.ext[1] ? 1 : 2);
  const int64_t delta = e - (ax == 0 ? 0 : ax == 1 ? g.ext[0] : g.ext[0] + g.ext[1]);
  const double dd = axis_distance(g, ax, 0, delta) * g.inv_c[ax];
  pc.d2tab[e] = dd * dd;
}

void launch_prepare(const ProblemTable& tab, ProblemDev* dtab, cudaStream_t st) {
  for (int first = 0; first < tab.count; first += kChunk) {
    TableChunk c;
    c.first = first;
    c.count = tab.count - first < kChunk ? tab.count - first : kChunk;
    int64_t emax = 1;
    for (int i = 0; i < c.count; ++i) {
      c.p[i] = tab.p[first + i];
      const GridDev& g = tab.p[first + i].grid;
      emax = std::max<int64_t>(emax, g.ext[0] + g.ext[1] + g.ext[2]);
    }
    k_prepare<<<dim3((unsigned)((emax + kPrepThreads - 1) / kPrepThreads), (unsigned)c.count), kPrepThreads, 0, st>>>(c, dtab);
    note_launches(1);
  }
}

// ---------------------------------------------------------------------------
// a1: ensemble mean and normalized anomalies Z (Eq. normalized_perturbations)
// ---------------------------------------------------------------------------
// One CTA per 32 consecutive state points (kAnomPts); warp w of the 8 takes
// the members w, w + 8, ...  Reads of X are coalesced over the points, the
// member sum is FP64 in a fixed order (per warp, then over the warps), and
// Z^T [n][N] is written through a shared-memory transpose, 32 members at a
// time, so that each point's member run is contiguous.
constexpr int kAnomPts = 32;
template <typename T>
__global__ void __launch_bounds__(256) k_anomalies(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.y];
  const int64_t x0 = (int64_t)blockIdx.x * kAnomPts;
  if (x0 >= pr.n) return;
  const int64_t N = pr.N, n = pr.n;
  const int lx = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t x = x0 + lx;
  const bool in = x < n;
  __shared__ double s_part[8][kAnomPts];
  __shared__ double s_mu[kAnomPts];
  __shared__ T s_tile[kAnomPts][33];
  __shared__ int s_bad;
  if (threadIdx.x == 0) s_bad = 0;
  double sum = 0.0;
  bool bad = false;
  if (in)
    for (int64_t k = w; k < N; k += 8) {
      const double v = pr.X[k * n + x];
      bad |= !isfinite(v);
      sum += v;
    }
  s_part[w][lx] = sum;
  __syncthreads();
  if (bad) s_bad = 1;
  if (w == 0) {
    double t = 0.0;
    for (int u = 0; u < 8; ++u) t += s_part[u][lx];
    const double mu = t / (double)N;
    s_mu[lx] = mu;
    if (in) pr.mu[x] = mu;
  }
  __syncthreads();
  const double mu = s_mu[lx];
  const double scale = 1.0 / pr.sqrt_nm1;
  T* Zt = tp<T>(pr.Zt);
  const int np = (int)(n - x0 < kAnomPts ? n - x0 : kAnomPts);
  for (int64_t c0 = 0; c0 < N; c0 += 32) {
    const int nk = (int)(N - c0 < 32 ? N - c0 : 32);
    for (int kk = w; kk < nk; kk += 8)
      s_tile[lx][kk] = in ? to_t<T>((pr.X[(c0 + kk) * n + x] - mu) * scale) : to_t<T>(0.0);
    __syncthreads();
    for (int e = threadIdx.x; e < np * 32; e += blockDim.x) {
      const int xi = e >> 5, kk = e & 31;
      if (kk < nk) Zt[(x0 + xi) * N + c0 + kk] = s_tile[xi][kk];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0 && s_bad) atomicOr(&pr.status[0], kStatNonFinite);
}

// W = H Z (rows of Z at the observed points), one thread per (observation,
// member) element so that the copy is coalesced; the member-0 thread of each
// observation also checks its index, forms R^-1/2 and the mean right-hand side.
template <typename T>
__global__ void k_observe(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.y];
  if (pr.H_rowptr) return;   // general observation operator: k_observe_H
  const int64_t N = pr.N;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= pr.d * N) return;
  const int64_t a = i / N, k = i - a * N;
  int64_t o = pr.obs[a];
  const bool bad_obs = o < 0 || o >= pr.n || (a > 0 && pr.obs[a - 1] >= o);
  if (o < 0) o = 0;
  if (o >= pr.n) o = pr.n - 1;
  tp<T>(pr.W)[i] = tp<const T>(pr.Zt)[o * N + k];
  if (k != 0) return;
  const double r = pr.R[a];
  const bool bad_r = !(r > 0.0) || !isfinite(r);
  const double ri = bad_r ? 0.0 : 1.0 / sqrt(r);
  pr.rinv[a] = ri;
  if (pr.do_mean) pr.bmean[a] = ri * (pr.y[a] - pr.mu[o]);
  if (bad_obs) atomicOr(&pr.status[0], kStatBadObs);
  if (bad_r) atomicOr(&pr.status[0], kStatBadR);
}

// ---------------------------------------------------------------------------
// General linear observation operator H (CSR, one row per observation; the
// paper's weighted sums, Sec. 4.1 and Sec. 5.1).  With h linearized and
// model-space localization (Sec. 2.3): W = H Z, Sxh = (L o Z Z^T) H^T,
// Shh = H Sxh, so C = R^-1/2 H Sxh R^-1/2.  Both are dense ([n][d], [d][d])
// and stored in the ELL layouts of the subsampling path with every column
// present, so the later stages run unchanged.  Row pointers and columns are
// checked before any entry is read.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool h_row(const ProblemDev& pr, int64_t a, int64_t& e0, int64_t& e1) {
  e0 = pr.H_rowptr[a];
  e1 = pr.H_rowptr[a + 1];
  if (e0 < 0 || e1 < e0 || e1 > pr.H_nnz || (a == 0 && e0 != 0)) {
    e0 = 0;
    e1 = 0;
    return false;
  }
  return true;
}

// W = H Z, one CTA per observation: its warps take the row's entries in turn,
// lanes over members (coalesced rows of Z^T), and the warps' sums are added in
// order; then R^-1/2 and the mean right-hand side R^-1/2 (y - H mu).  (One
// thread per (observation, member) walked the whole row: 67 us at 100 rows of
// 137 entries, on eight SMs.)
constexpr int kHWarps = 8;
template <typename T>
__global__ void __launch_bounds__(32 * kHWarps) k_observe_H(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.y];
  if (!pr.H_rowptr) return;
  const int64_t a = blockIdx.x, N = pr.N;
  if (a >= pr.d) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ double part[kHWarps][32];
  __shared__ double mpart[kHWarps];
  __shared__ int s_bad;
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  int64_t e0, e1;
  bool bad = !h_row(pr, a, e0, e1);
  const T* Zt = tp<const T>(pr.Zt);
  double hmu = 0.0;
  for (int64_t k0 = 0; k0 < N; k0 += 32) {
    const int64_t k = k0 + lane;
    double w = 0.0;
#pragma unroll 4
    for (int64_t e = e0 + warp; e < e1; e += kHWarps) {
      const int64_t c = pr.H_col[e];
      if (c < 0 || c >= pr.n) {
        bad = true;
        continue;
      }
      const double h = pr.H_val[e];
      if (k < N) w += h * (double)Zt[c * N + k];
      if (k == 0) hmu += h * pr.mu[c];
    }
    part[warp][lane] = w;
    if (k == 0) mpart[warp] = hmu;
    __syncthreads();
    if (warp == 0 && k < N) {
      double t = 0.0;
#pragma unroll
      for (int u = 0; u < kHWarps; ++u) t += part[u][lane];
      tp<T>(pr.W)[a * N + k] = to_t<T>(t);
    }
    __syncthreads();
  }
  if (bad) s_bad = 1;
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int u = 1; u < kHWarps; ++u) hmu += mpart[u];   // thread 0 holds warp 0's sum
  const double r = pr.R[a];
  const bool bad_r = !(r > 0.0) || !isfinite(r);
  const double ri = bad_r ? 0.0 : 1.0 / sqrt(r);
  pr.rinv[a] = ri;
  if (pr.do_mean) pr.bmean[a] = ri * (pr.y[a] - hmu);
  if (s_bad) atomicOr(&pr.status[0], kStatBadObs);
  if (bad_r) atomicOr(&pr.status[0], kStatBadR);
}

// Sxh(x, b) = sum_j H(b, j) L(x, j) z_x . z_j.  A CTA owns kXB consecutive grid
// points: it forms their rows G_x(j) = L(x, j) z_x . z_j over all grid points
// once in shared memory (zero outside the support), then takes H G_x^T row by
// row, one warp per observation with its lanes over the row's entries; rows
// that miss the supports cost no arithmetic.  (Each (x, b) formed its own
// products z_x . z_j, so every pair (x, j) was formed once per observation
// that sees j: 656 to 865 us at n = 2000, d = 100, rows of 137 entries; 155 us with
// the squared distance of every pair in FP64, 115 us with the support's box checked in integers.)
constexpr int kXB = 4;
constexpr size_t kSxhSmem = 200 * 1024;
template <typename T>
__global__ void __launch_bounds__(256) k_sxh_H(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.y];
  if (!pr.H_rowptr) return;
  extern __shared__ double Gx[];   // [n][kXB]
  const int64_t n = pr.n, N = pr.N, d = pr.d;
  const int64_t x0 = (int64_t)blockIdx.x * kXB;
  if (x0 >= n || (size_t)n * kXB * 8 > kSxhSmem) return;   // larger grids: k_sxh_H_direct
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const GridDev& g = pr.grid;
  const T* Zt = tp<const T>(pr.Zt);
  Coord3 px[kXB];
#pragma unroll
  for (int u = 0; u < kXB; ++u) px[u] = flat_to_coord32(g, (uint32_t)(x0 + u < n ? x0 + u : x0));
  // in integers: beyond the support's box on some axis
  auto outside = [&](const Coord3& a, const Coord3& b) {
    const int64_t ca[3] = {a.x, a.y, a.z}, cb[3] = {b.x, b.y, b.z};
    bool out = false;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      if (g.whole[ax]) continue;
      int64_t delta = ca[ax] > cb[ax] ? ca[ax] - cb[ax] : cb[ax] - ca[ax];
      if (g.periodic[ax] && g.ext[ax] - delta < delta) delta = g.ext[ax] - delta;
      out |= delta > g.reach[ax];
    }
    return out;
  };
  for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
    const Coord3 pj = flat_to_coord32(g, (uint32_t)j);
    const T* zj = Zt + j * N;
    for (int u = 0; u < kXB; ++u) {
      double v = 0.0;
      if (x0 + u < n && !outside(px[u], pj)) {
        const double r2 = scaled_r2_tab(g, pr.d2tab, px[u], pj);
        if (r2 < 4.0) {
          DotAcc<T> dot;
          const T* zx = Zt + (x0 + u) * N;
          for (int64_t k = 0; k < N; ++k) dot.add_prod(zx[k], zj[k]);
          const double gc = sizeof(T) == 8 ? gaspari_cohn(sqrt(r2)) : (double)gaspari_cohn_f(sqrtf((float)r2));
          v = gc * dot.value();
        }
      }
      Gx[j * kXB + u] = v;
    }
  }
  __syncthreads();
  for (int64_t b = warp; b < d; b += nw) {
    int64_t e0, e1;
    h_row(pr, b, e0, e1);
    double acc[kXB] = {};
    bool hit = false;
    for (int64_t e = e0 + lane; e < e1; e += 32) {
      const int64_t c = pr.H_col[e];
      if (c < 0 || c >= n) continue;
      const double* gx = Gx + c * kXB;
      bool any = false;
#pragma unroll
      for (int u = 0; u < kXB; ++u) any |= __double_as_longlong(gx[u]) != 0;
      if (!any) continue;
      hit = true;
      const double h = pr.H_val[e];
#pragma unroll
      for (int u = 0; u < kXB; ++u) acc[u] += h * gx[u];
    }
    if (__any_sync(0xffffffffu, hit)) {
#pragma unroll
      for (int u = 0; u < kXB; ++u) acc[u] = warp_sum(acc[u]);
    }
    if (lane < kXB && x0 + lane < n) {
      double v = acc[0];
#pragma unroll
      for (int u = 1; u < kXB; ++u) v = lane == u ? acc[u] : v;
      tp<T>(pr.xo_val)[b * n + x0 + lane] = to_t<T>(v);
      pr.xo_col[b * n + x0 + lane] = (int32_t)b;
      if (b == 0) pr.xo_nnz[x0 + lane] = (int32_t)d;
    }
  }
}

// The same for grids whose rows do not fit shared memory: thread x
// (consecutive, so that the ELL writes are coalesced) of observation column
// b = blockIdx.y forms its own products.
template <typename T>
__global__ void k_sxh_H_direct(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.z];
  if (!pr.H_rowptr || (size_t)pr.n * kXB * 8 <= kSxhSmem) return;
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t b = blockIdx.y;
  const int64_t n = pr.n, N = pr.N;
  if (x >= n || b >= pr.d) return;
  const GridDev& g = pr.grid;
  const Coord3 px = flat_to_coord(g, x);
  const T* Zt = tp<const T>(pr.Zt);
  const T* zx = Zt + x * N;
  int64_t e0, e1;
  h_row(pr, b, e0, e1);
  double acc = 0.0;
  for (int64_t e = e0; e < e1; ++e) {
    const int64_t c = pr.H_col[e];
    if (c < 0 || c >= n) continue;
    const double r2 = scaled_r2_tab(g, pr.d2tab, px, flat_to_coord(g, c));
    if (!(r2 < 4.0)) continue;
    DotAcc<T> dot;
    const T* zc = Zt + c * N;
    for (int64_t k = 0; k < N; ++k) dot.add_prod(zx[k], zc[k]);
    const double gc = sizeof(T) == 8 ? gaspari_cohn(sqrt(r2)) : (double)gaspari_cohn_f(sqrtf((float)r2));
    acc += pr.H_val[e] * gc * dot.value();
  }
  tp<T>(pr.xo_val)[b * n + x] = to_t<T>(acc);
  pr.xo_col[b * n + x] = (int32_t)b;
  if (b == 0) pr.xo_nnz[x] = (int32_t)pr.d;
}

// C(a, b) = R_a^-1/2 R_b^-1/2 sum_x H(a, x) Sxh(x, b), one CTA per row a: a warp
// per entry with its lanes over the row of H (a column of Sxh is contiguous);
// the Gershgorin bound, the minimum and the sum of the diagonal as in k_band.
template <typename T>
__global__ void __launch_bounds__(32 * kHWarps) k_c_H(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.y];
  if (!pr.H_rowptr) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t a = blockIdx.x, n = pr.n, d = pr.d;
  if (a >= d) return;
  __shared__ double part[kHWarps];
  int64_t e0, e1;
  h_row(pr, a, e0, e1);
  const T* S = tp<const T>(pr.xo_val);
  const double ra = pr.rinv[a];
  double rowsum = 0.0;
  for (int64_t b = warp; b < d; b += kHWarps) {
    double acc = 0.0;
    for (int64_t e = e0 + lane; e < e1; e += 32) {
      const int64_t c = pr.H_col[e];
      if (c < 0 || c >= n) continue;
      acc += pr.H_val[e] * (double)S[b * n + c];
    }
    acc = warp_sum(acc);
    if (lane != 0) continue;
    const double v = ra * pr.rinv[b] * acc;
    tp<T>(pr.oo_val)[b * d + a] = to_t<T>(v);
    pr.oo_col[b * d + a] = (int32_t)b;
    rowsum += fabs(v);
    if (b == a) {
      atomic_min_nonneg(&pr.scal[1], fmax(v, 0.0));
      atomicAdd(&pr.scal[4], v);
    }
  }
  if (lane == 0) part[warp] = rowsum;
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int u = 1; u < kHWarps; ++u) rowsum += part[u];
  pr.oo_nnz[a] = (int32_t)d;
  atomic_max_nonneg(&pr.scal[0], rowsum);
}

void launch_anomalies(const ProblemTable& tab, const ProblemDev* dtab, cudaStream_t st) {
  int64_t nmax = 0, dnmax = 0, dh = 0;   // dh: most observations of a general H
  for (int i = 0; i < tab.count; ++i) {
    if (tab.p[i].H_rowptr) dh = std::max<int64_t>(dh, tab.p[i].d);
    nmax = tab.p[i].n > nmax ? tab.p[i].n : nmax;
    dnmax = tab.p[i].d * tab.p[i].N > dnmax ? tab.p[i].d * tab.p[i].N : dnmax;
  }
  const bool f64 = tab.p[0].precision == 0;
  dim3 g1((unsigned)((nmax + kAnomPts - 1) / kAnomPts), tab.count);
  dim3 g2((unsigned)((dnmax + 255) / 256), tab.count);
  const dim3 gh((unsigned)dh, tab.count);
  if (f64) {
    k_anomalies<double><<<g1, 256, 0, st>>>(dtab); note_launches(1);
    k_observe<double><<<g2, 256, 0, st>>>(dtab); note_launches(1);
    if (dh > 0) { k_observe_H<double><<<gh, 32 * kHWarps, 0, st>>>(dtab); note_launches(1); }
  } else {
    k_anomalies<float><<<g1, 256, 0, st>>>(dtab); note_launches(1);
    k_observe<float><<<g2, 256, 0, st>>>(dtab); note_launches(1);
    if (dh > 0) { k_observe_H<float><<<gh, 32 * kHWarps, 0, st>>>(dtab); note_launches(1); }
  }
}

// ---------------------------------------------------------------------------
// Bands.  One warp per row.  Lanes take consecutive candidate obs b from the
// geometry's candidate ranges, keep those with r < 2, and append
//   C(a, b) = GC(r) (w_a . w_b) R_a^-1/2 R_b^-1/2        (obs-obs, rows = obs)
//   Sxh(x, b) = GC(r) (z_x . w_b)                        (state-obs, rows = state)
// in increasing candidate order to the ELL row (column-major: entry e of row
// a at e * rows + a).  Two warps per CTA, so that small problems spread over all
// SMs (an FP64 instruction of a warp holds its SM's pipe for 16 clocks); candidates
// found by the whole warp, 32-bit coordinates.  8192 points and 1024 observations
// FP32: 72 -> 52 us (state rows) and 26 -> 20 us; 240 and 60 FP64: 17 -> 12 and 18 -> 13 us.
// ---------------------------------------------------------------------------
constexpr int kBandThreads = 64;
template <typename T, bool OBS_ROWS>
__global__ void __launch_bounds__(kBandThreads) k_band(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.y];
  if (pr.H_rowptr) return;   // general observation operator: k_sxh_H and k_c_H
  const int lane = threadIdx.x & 31;
  const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t rows = OBS_ROWS ? pr.d : pr.n;
  if (row >= rows) return;
  const int64_t N = pr.N, d = pr.d;
  const GridDev& g = pr.grid;
  int64_t pidx = OBS_ROWS ? pr.obs[row] : row;
  if (pidx < 0) pidx = 0;
  if (pidx >= pr.n) pidx = pr.n - 1;
  const Coord3 pc = flat_to_coord32(g, (uint32_t)pidx);   // n < 2^31 (checked by the host)
  const T* W = tp<const T>(pr.W);
  const T* src = OBS_ROWS ? W + row * N : tp<const T>(pr.Zt) + row * N;
  const int64_t cap = OBS_ROWS ? pr.max_oo : pr.max_xo;
  T* val = OBS_ROWS ? tp<T>(pr.oo_val) : tp<T>(pr.xo_val);
  int32_t* col = OBS_ROWS ? pr.oo_col : pr.xo_col;
  const double ra = OBS_ROWS ? pr.rinv[row] : 1.0;
  int64_t count = 0;
  double rowsum = 0.0;
  for_each_candidate_range<true>(g, pr.obs, d, pc, [&](int64_t b0, int64_t b1) {
    for (int64_t base = b0; base < b1; base += 32) {
      const int64_t b = base + lane;
      double v = 0.0;
      bool keep = false;
      const int64_t ib = b < b1 ? pr.obs[b] : -1;
      if (ib >= 0 && ib < pr.n) {
        const Coord3 bc = flat_to_coord32(g, (uint32_t)ib);
        const double r2 = scaled_r2_tab(g, pr.d2tab, pc, bc);
        if (r2 < 4.0) {
          keep = true;
          DotAcc<T> acc;
          const T* wb = W + b * N;
          // 16-byte loads when the member rows allow them (same order of terms)
          if (sizeof(T) == 4 && (N & 3) == 0) {
            const float4* s4 = reinterpret_cast<const float4*>(src);
            const float4* w4 = reinterpret_cast<const float4*>(wb);
            for (int64_t k = 0; k < N / 4; ++k) {
              const float4 u = s4[k], v4 = w4[k];
              acc.add_prod((T)u.x, (T)v4.x);
              acc.add_prod((T)u.y, (T)v4.y);
              acc.add_prod((T)u.z, (T)v4.z);
              acc.add_prod((T)u.w, (T)v4.w);
            }
          } else if (sizeof(T) == 8 && (N & 1) == 0) {
            const double2* s2 = reinterpret_cast<const double2*>(src);
            const double2* w2 = reinterpret_cast<const double2*>(wb);
            for (int64_t k = 0; k < N / 2; ++k) {
              const double2 u = s2[k], v2 = w2[k];
              acc.add_prod((T)u.x, (T)v2.x);
              acc.add_prod((T)u.y, (T)v2.y);
            }
          } else {
            for (int64_t k = 0; k < N; ++k) acc.add_prod(src[k], wb[k]);
          }
          const double gc = sizeof(T) == 8 ? gaspari_cohn(sqrt(r2)) : (double)gaspari_cohn_f(sqrtf((float)r2));
          v = gc * acc.value();
          if (OBS_ROWS) v *= ra * pr.rinv[b];
        }
      }
      const unsigned mask = __ballot_sync(0xffffffffu, keep);
      const int before = __popc(mask & ((1u << lane) - 1u));
      if (keep) {
        const int64_t e = count + before;
        if (e < cap) {
          val[e * rows + row] = to_t<T>(v);
          col[e * rows + row] = (int32_t)b;
        }
        if (OBS_ROWS) rowsum += fabs(v);
        if (OBS_ROWS && b == row) {
          atomic_min_nonneg(&pr.scal[1], v);
          atomicAdd(&pr.scal[4], v);
        }
      }
      count += __popc(mask);
    }
  });
  if (OBS_ROWS) rowsum = warp_sum(rowsum);
  if (lane == 0) {
    int32_t* nnz = OBS_ROWS ? pr.oo_nnz : pr.xo_nnz;
    nnz[row] = (int32_t)(count < cap ? count : cap);
    if (count > cap) atomicOr(&pr.status[0], kStatBandOverflow);
    if (OBS_ROWS) atomic_max_nonneg(&pr.scal[0], rowsum);
  }
}

// Band of C (obs rows); the distance table comes from launch_prepare.
void launch_band_obs(const ProblemTable& tab, const ProblemDev* dtab, cudaStream_t st) {
  int64_t dmax = 0;
  for (int i = 0; i < tab.count; ++i) dmax = tab.p[i].d > dmax ? tab.p[i].d : dmax;
  dim3 go((unsigned)((dmax * 32 + kBandThreads - 1) / kBandThreads), tab.count);
  if (tab.p[0].precision == 0) k_band<double, true><<<go, kBandThreads, 0, st>>>(dtab);
  else k_band<float, true><<<go, kBandThreads, 0, st>>>(dtab);
  note_launches(1);
  int64_t dh = 0;   // most observations of a general H
  for (int i = 0; i < tab.count; ++i)
    if (tab.p[i].H_rowptr) dh = std::max<int64_t>(dh, tab.p[i].d);
  if (dh > 0) {
    // dense Sxh first (C is formed from it), then C
    // grids whose rows of L o Z Z^T fit shared memory, then the others
    const size_t row = (size_t)kXB * 8;
    int64_t nfit = 0, nbig = 0;
    for (int i = 0; i < tab.count; ++i)
      if (tab.p[i].H_rowptr) {
        int64_t& most = (size_t)tab.p[i].n * row <= kSxhSmem ? nfit : nbig;
        most = std::max<int64_t>(most, tab.p[i].n);
      }
    const bool f64 = tab.p[0].precision == 0;
    if (nfit > 0) {
      const dim3 gs((unsigned)((nfit + kXB - 1) / kXB), tab.count);
      const size_t smem = (size_t)nfit * row;
      static thread_local int raised = -1;
      int dev = 0;
      cudaGetDevice(&dev);
      if (raised != dev) {
        cudaFuncSetAttribute(k_sxh_H<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSxhSmem);
        cudaFuncSetAttribute(k_sxh_H<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSxhSmem);
        raised = dev;
      }
      if (f64) k_sxh_H<double><<<gs, 256, smem, st>>>(dtab);
      else k_sxh_H<float><<<gs, 256, smem, st>>>(dtab);
      note_launches(1);
    }
    if (nbig > 0) {
      const dim3 gs((unsigned)((nbig + 127) / 128), (unsigned)dh, tab.count);
      if (f64) k_sxh_H_direct<double><<<gs, 128, 0, st>>>(dtab);
      else k_sxh_H_direct<float><<<gs, 128, 0, st>>>(dtab);
      note_launches(1);
    }
    const dim3 gc((unsigned)dh, tab.count);
    if (f64) k_c_H<double><<<gc, 32 * kHWarps, 0, st>>>(dtab);
    else k_c_H<float><<<gc, 32 * kHWarps, 0, st>>>(dtab);
    note_launches(1);
  }
}

// Band of Sxh (state rows); needed only by the state update.
void launch_band_state(const ProblemTable& tab, const ProblemDev* dtab, cudaStream_t st) {
  int64_t nmax = 0;
  for (int i = 0; i < tab.count; ++i) nmax = tab.p[i].n > nmax ? tab.p[i].n : nmax;
  dim3 gx((unsigned)((nmax * 32 + kBandThreads - 1) / kBandThreads), tab.count);
  if (tab.p[0].precision == 0) k_band<double, false><<<gx, kBandThreads, 0, st>>>(dtab);
  else k_band<float, false><<<gx, kBandThreads, 0, st>>>(dtab);
  note_launches(1);
}

void launch_bands(const ProblemTable& tab, const ProblemDev* dtab, cudaStream_t st) {
  launch_band_obs(tab, dtab, st);
  launch_band_state(tab, dtab, st);
}

// Counts neighbours to size the bands: out2[0] = max obs per obs row,
// out2[1] = max obs per state row.
__global__ void k_count_neighbours(const GridDev g, const int64_t* obs, int64_t d, int64_t n,
                                   unsigned long long* out2) {
  const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= n + d) return;
  const bool is_obs = row >= n;
  int64_t pidx = is_obs ? obs[row - n] : row;
  if (pidx < 0) pidx = 0;
  if (pidx >= n) pidx = n - 1;
  const Coord3 pc = flat_to_coord(g, pidx);
  unsigned long long count = 0;
  for_each_candidate_range(g, obs, d, pc, [&](int64_t b0, int64_t b1) {
    for (int64_t b = b0; b < b1; ++b) {
      if (scaled_distance(g, pc, flat_to_coord(g, obs[b])) < 2.0) ++count;
    }
  });
  atomicMax(&out2[is_obs ? 0 : 1], count);
}

void launch_count_neighbours(const GridDev& g, const int64_t* obs, int64_t d, int64_t n,
                             int64_t* out2, cudaStream_t st) {
  cudaMemsetAsync(out2, 0, 2 * sizeof(int64_t), st);
  const int64_t rows = n + d;
  k_count_neighbours<<<(unsigned)((rows + 255) / 256), 256, 0, st>>>(
      g, obs, d, n, reinterpret_cast<unsigned long long*>(out2));
  note_launches(1);
}

// ---------------------------------------------------------------------------
// a2: quadrature (App. D).  Elliptic rule with modulus g = sqrt(ell/(1+ell)):
//   s_q = sc(u_q | g)^2,  p_q = (2 K / (pi Q)) dn(u_q | g),  u_q = (q - 1/2) K / Q,
// which is r_q / (s_q + 1) with r_q = (2K/(pi Q)) nc dc (d sc/du = dc nc and
// sc^2 + 1 = nc^2).  K and the Jacobi functions come from one descending
// Landen ladder in float-float (quadrature_node); nodes past K/2 use
// sn(K - v) = cd(v), cn(K - v) = g' sd(v), dn(K - v) = g' nd(v) so that small
// cn values keep full relative precision.
// ---------------------------------------------------------------------------
// pi / 2 as a float-float pair, and the Taylor coefficients (-1)^j / (2j+1)! and
// (-1)^j / (2j)!, j = 0..9, as exact float-float pairs (hexadecimal literals).
constexpr float kPiHalfHi = 0x1.921fb6p+0f, kPiHalfLo = -0x1.777a5cp-25f;
__constant__ float kSinH[10] = {0x1p+0f, -0x1.555556p-3f, 0x1.111112p-7f, -0x1.a01a02p-13f, 0x1.71de3ap-19f,
                                -0x1.ae6456p-26f, 0x1.612462p-33f, -0x1.ae7f3ep-41f, 0x1.952c78p-49f,
                                -0x1.2f49b4p-57f};
__constant__ float kSinL[10] = {0.f, 0x1.555556p-28f, -0x1.dddddep-32f, 0x1.7f97fap-39f, 0x1.55b1ccp-45f,
                                -0x1.fd5138p-52f, -0x1.8af25ep-58f, -0x1.ccee08p-67f, -0x1.f9ea56p-74f,
                                -0x1.a05056p-83f};
__constant__ float kCosH[10] = {0x1p+0f, -0x1p-1f, 0x1.555556p-5f, -0x1.6c16c2p-10f, 0x1.a01a02p-16f,
                                -0x1.27e4fcp-22f, 0x1.1eed8ep-29f, -0x1.93974ap-37f, 0x1.ae7f3ep-45f,
                                -0x1.682786p-53f};
__constant__ float kCosL[10] = {0.f, 0.f, -0x1.555556p-30f, 0x1.27d27ep-35f, -0x1.7f97fap-42f, 0x1.10ec14p-47f,
                                0x1.ff1b14p-54f, -0x1.180f94p-62f, 0x1.ccee08p-71f, -0x1.dcbeccp-80f};

// sin x and cos x for |x| <= pi/4 in float-float: Taylor series by Horner's
// rule in x^2, truncated after x^19 (sin) and x^18 (cos), below 1e-17 there.
__device__ void ff_sincos_small(FF x, FF& sn, FF& cn) {
  const FF x2 = ff_mul(x, x);
  FF as{kSinH[9], kSinL[9]}, ac{kCosH[9], kCosL[9]};
  for (int j = 8; j >= 0; --j) {
    as = ff_add(FF{kSinH[j], kSinL[j]}, ff_mul(as, x2));
    ac = ff_add(FF{kCosH[j], kCosL[j]}, ff_mul(ac, x2));
  }
  sn = ff_mul(x, as);
  cn = ac;
}

__device__ void quadrature_node(int32_t Q, double ell, int32_t rule, int q, double& s, double& p) {
  if (rule == 1) {
    // Gauss-Legendre on (0,1) for the trigonometric form (Eq. gaussian_quadrature_rule);
    // Newton iteration on P_Q with the three-term recurrence.
    double x = cos(kPi * (q + 0.75) / (Q + 0.5));
    double dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = x;
      for (int k = 2; k <= Q; ++k) {
        const double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      if (Q == 1) { p1 = x; p0 = 1.0; }
      dp = Q * (x * p1 - p0) / (x * x - 1.0);
      const double dx = p1 / dp;
      x -= dx;
      if (fabs(dx) < 1e-16) {
        break;
      }
    }
    {
      double p0 = 1.0, p1 = x;
      for (int k = 2; k <= Q; ++k) {
        const double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = Q * (x * p1 - p0) / (x * x - 1.0);
    }
    const double v = 2.0 / ((1.0 - x * x) * dp * dp);
    const double lam = 0.5 * (1.0 - x);   // ascending order in q
    const double tn = tan(0.5 * kPi * lam);
    s = tn * tn;
    p = 0.5 * v;
    return;
  }
  // Elliptic rule in float-float (about 48 bits, FP32 instructions only; a
  // chain of FP64 instructions is slow on this GPU).  Descending Landen
  // ladder of the modulus g (g^2 = ell / (1 + ell), g' = (1 + ell)^-1/2):
  //   k_{n+1} = k_n^2 / (1 + k'_n)^2 = (1 - k'_n) / (1 + k'_n),  k'_{n+1} = 2 sqrt(k'_n) / (1 + k'_n),
  // free of cancellation for k near 1, with K = (pi/2) prod_n (1 + k_n).  The
  // argument at the bottom of the ladder is u prod_n (1 + k_n)^-1 = t pi / 2
  // for u = t K, so sin and cos are of a known angle <= pi/4 (Taylor series);
  // sn, cn, dn then ascend the ladder by the descending Landen (Gauss)
  // transformation (Abramowitz & Stegun 16.12): with s2 = k_{n+1} sn^2,
  //   sn <- (1 + k_{n+1}) sn / (1 + s2),  cn <- cn dn / (1 + s2),  dn <- (1 - s2) / (1 + s2).
  // Nodes past K/2 use the reflection below.
  const FF one{1.f, 0.f};
  const FF L = ff_from(ell);
  const FF kp0 = ff_rsqrt(ff_add(one, L));
  FF k = ff_mul(ff_sqrt(L), kp0), kp = kp0, prod = one;
  FF ks[24];
  int nk = 0;
  while (k.h > 1e-17f && nk < 24) {
    const FF opk = ff_add(one, kp);
    const FF k1 = ff_div(ff_mul(k, k), ff_mul(opk, opk));
    ks[nk++] = k1;
    prod = ff_mul(prod, ff_add(one, k1));
    kp = ff_div(ff_mul(FF{2.f, 0.f}, ff_sqrt(kp)), opk);
    k = k1;
  }
  const double t = (q + 0.5) / Q;
  const bool refl = t > 0.5;
  const double tt = refl ? ((Q - q) - 0.5) / Q : t;   // K - u_q, formed without cancellation
  FF sn, cn;
  ff_sincos_small(ff_mul(FF{kPiHalfHi, kPiHalfLo}, ff_from(tt)), sn, cn);
  FF dn = one;
  for (int i = nk - 1; i >= 0; --i) {
    const FF s2 = ff_mul(ks[i], ff_mul(sn, sn));
    const FF den = ff_div(one, ff_add(one, s2));
    const FF s_new = ff_mul(ff_mul(ff_add(one, ks[i]), sn), den);
    const FF c_new = ff_mul(ff_mul(cn, dn), den);
    dn = ff_mul(ff_sub(one, s2), den);
    sn = s_new;
    cn = c_new;
  }
  const FF scale = ff_div(prod, ff_from((double)Q));   // 2 K / (pi Q)
  FF sq, pq;
  if (!refl) {
    const FF r = ff_div(sn, cn);                       // sc(u_q)
    sq = ff_mul(r, r);
    pq = ff_mul(scale, dn);
  } else {
    const FF r = ff_div(cn, ff_mul(kp0, sn));          // sc(K - v) = cd(v) / (g' sd(v))
    sq = ff_mul(r, r);
    pq = ff_div(ff_mul(scale, kp0), dn);               // dn(K - v) = g' / dn(v)
  }
  s = (double)sq.h + (double)sq.l;
  p = (double)pq.h + (double)pq.l;
}

__global__ void k_quadrature(ProblemDev* tab) {
  ProblemDev& pr = tab[blockIdx.x];
  __shared__ double ell_s;
  if (threadIdx.x == 0) {
    double ell = pr.ell_fixed;
    if (!(ell > 0.0)) {
      const double b = fmax(pr.scal[0], 1.0);
      ell = exp10(floor(log10(b)) + 1.0);
    }
    ell_s = ell;
    pr.scal[2] = ell;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < pr.Q; q += blockDim.x) {
    double s, p;
    quadrature_node(pr.Q, ell_s, pr.rule, q, s, p);
    pr.s[q] = s;
    pr.p[q] = p;
  }
}

void launch_quadrature(const ProblemTable& tab, const ProblemDev* dtab, cudaStream_t st) {
  k_quadrature<<<tab.count, 64, 0, st>>>(const_cast<ProblemDev*>(dtab)); note_launches(1);
}

__global__ void k_quadrature_nodes(int32_t Q, double ell, int32_t rule, double* s, double* p) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < Q) quadrature_node(Q, ell, rule, q, s[q], p[q]);
}

void launch_quadrature_nodes(int32_t Q, double ell, int32_t rule, double* s, double* p, cudaStream_t st) {
  k_quadrature_nodes<<<(Q + 63) / 64, 64, 0, st>>>(Q, ell, rule, s, p); note_launches(1);
}

__global__ void k_philox(uint64_t seed, int64_t count, double* out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < count) out[e] = philox_normal(seed, (uint64_t)e);
}

void launch_philox(uint64_t seed, int64_t count, double* out, cudaStream_t st) {
  if (count > 0) {
    k_philox<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(seed, count, out);
    note_launches(1);
  }
}

// ---------------------------------------------------------------------------
// a4: randomized Ritz pairs of C (App. E; Halko, Martinsson, Tropp Alg. 5.3
// on a range basis from their Alg. 4.3 with power_iters power iterations).
//
// Two [d][l] buffers of the bulk type T (Om and Yb) hold the basis and its
// image under C; `src` selects which one a kernel reads.  Gram matrices are
// summed with DotAcc<T> and kept in FP64.  Orthonormalization is CholeskyQR2
// (each pass: G = X^T X, G = R^T R, X <- X R^-1, the Cholesky factor formed
// redundantly by every row block).  The l x l eigenproblem uses cyclic
// Jacobi with l/2 disjoint rotations per round (round-robin ordering) in
// FP32, refined by products on the FP64 path.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T* ritz_buf(const ProblemDev& pr, int which) {
  return reinterpret_cast<T*>(which == 0 ? pr.Om : pr.Yb);
}

template <typename T>
__global__ void k_ritz_omega(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.y];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (pr.l <= 0 || i >= pr.d * pr.l) return;
  const int64_t a = i / pr.l, j = i % pr.l;
  ritz_buf<T>(pr, 0)[i] = to_t<T>(philox_normal(pr.seed, (uint64_t)(j * pr.d + a)));
}

// dst = C src: one warp per row, lanes over the row's band entries; each lane
// accumulates all l columns of its entries, then a butterfly reduce-scatter
// leaves column j's sum in lane j.
template <typename T>
__global__ void k_ritz_matvec(const ProblemDev* tab, int src) {
  const ProblemDev& pr = tab[blockIdx.y];
  const int l = pr.l;
  const int lane = threadIdx.x & 31;
  const int64_t a = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (l <= 0 || a >= pr.d) return;
  const int64_t d = pr.d;
  const T* __restrict__ V = ritz_buf<T>(pr, src);
  T* Y = ritz_buf<T>(pr, 1 - src);
  const T* __restrict__ val = tp<const T>(pr.oo_val);
  const int32_t* __restrict__ col = pr.oo_col;
  const int nnz = pr.oo_nnz[a];
  T acc[32];
#pragma unroll
  for (int m = 0; m < 32; ++m) acc[m] = T(0);
  const bool vec4 = sizeof(T) == 4 && (l & 3) == 0;
  for (int e = lane; e < nnz; e += 32) {
    const T c = val[(int64_t)e * d + a];
    const T* vr = V + (int64_t)col[(int64_t)e * d + a] * l;
    if (vec4) {
#pragma unroll
      for (int m4 = 0; m4 < 8; ++m4) {
        if (4 * m4 < l) {
          const float4 v = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(vr) + 4 * m4);
          acc[4 * m4 + 0] += c * (T)v.x;
          acc[4 * m4 + 1] += c * (T)v.y;
          acc[4 * m4 + 2] += c * (T)v.z;
          acc[4 * m4 + 3] += c * (T)v.w;
        }
      }
    } else {
#pragma unroll
      for (int m = 0; m < 32; ++m)
        if (m < l) acc[m] += c * vr[m];
    }
  }
  const T sum = warp_reduce_scatter32<T>(acc, lane);
  if (lane < l) Y[a * l + lane] = sum;
}

// G[i][j] = sum_a A[a][i] B[a][j] (FP64 result), one block per entry.
// sym: A = B = buf(src) and only j >= i is computed (mirrored).
template <typename T>
__global__ void k_ritz_gram(const ProblemDev* tab, int srcA, int srcB, int sym) {
  const ProblemDev& pr = tab[blockIdx.y];
  const int l = pr.l;
  const int pair = blockIdx.x;
  if (l <= 0 || pair >= l * l) return;
  const int i = pair / l, j = pair % l;
  if (sym && j < i) return;
  const T* A = ritz_buf<T>(pr, srcA);
  const T* Bm = ritz_buf<T>(pr, srcB);
  DotAcc<T> acc;
  for (int64_t a = threadIdx.x; a < pr.d; a += blockDim.x) acc.add_prod(A[a * l + i], Bm[a * l + j]);
  DotAcc<T> accs[1] = {acc};
  double out[1];
  __shared__ double scratch[2 * kThreads / 32];
  block_sum<1>(accs, out, scratch);
  if (threadIdx.x == 0) {
    pr.Gm[i * l + j] = out[0];
    if (sym) pr.Gm[j * l + i] = out[0];
  }
}

// X_dst = X_src R^-1 with G = R^T R the Cholesky factorization of the Gram
// matrix in Gm.  Right-looking factorization in float-float arithmetic by four
// warps: warp 0 takes the pivot's reciprocal square root, all threads scale
// row j and update the trailing upper triangle.  A non-positive pivot zeroes
// that column (rank loss) and flags kStatEigFail.  R goes to shared memory in
// the bulk type for the triangular solve, one thread per row.
template <typename T>
__global__ void k_ritz_orth(const ProblemDev* tab, int src) {
  const ProblemDev& pr = tab[blockIdx.y];
  const int l = pr.l;
  if (l <= 0) return;
  __shared__ FF G[kMaxRitz][kMaxRitz + 1];
  __shared__ FF Rrow[kMaxRitz];
  __shared__ FF s_inv;
  __shared__ float s_tiny;
  __shared__ T Rt[kMaxRitz][kMaxRitz + 1];
  __shared__ T rinv[kMaxRitz];
  for (int e = threadIdx.x; e < l * l; e += blockDim.x) {
    const int i = e / l, c = e % l;
    if (i <= c) G[i][c] = ff_from(pr.Gm[e]);
  }
  if (threadIdx.x < 32) {
    float tr = threadIdx.x < l ? (float)pr.Gm[threadIdx.x * (l + 1)] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
    if (threadIdx.x == 0) s_tiny = 1e-28f * (tr > 0.f ? tr : 1.f);
  }
  __syncthreads();
  constexpr int kCT = 128;
  const int t = threadIdx.x;
  if (t < kCT) {
    const float tiny = s_tiny;
    for (int j = 0; j < l; ++j) {
      if (t == 0) {
        const FF gjj = G[j][j];
        const bool ok = gjj.h > tiny;
        const FF inv = ok ? ff_rsqrt(gjj) : FF{0.f, 0.f};
        s_inv = inv;
        const FF rjj = ff_mul(gjj, inv);
        Rt[j][j] = (T)rjj.h + (T)rjj.l;
        rinv[j] = (T)inv.h + (T)inv.l;
        if (!ok && blockIdx.x == 0) atomicOr(&pr.status[0], kStatEigFail);
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      const FF inv = s_inv;
      for (int c = j + 1 + t; c < l; c += kCT) {
        const FF r = ff_mul(G[j][c], inv);
        Rrow[c] = r;
        Rt[j][c] = (T)r.h + (T)r.l;
      }
      if (t < j) Rt[j][t] = T(0);
      asm volatile("bar.sync 1, 128;" ::: "memory");
      const int mrem = l - 1 - j;
      for (int e = t; e < mrem * mrem; e += kCT) {
        const int c2 = j + 1 + e / mrem, c = j + 1 + e % mrem;
        if (c2 <= c) G[c2][c] = ff_sub(G[c2][c], ff_mul(Rrow[c2], Rrow[c]));
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
    }
  }
  __syncthreads();
  const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= pr.d) return;
  const T* X = ritz_buf<T>(pr, src);
  T* Y = ritz_buf<T>(pr, 1 - src);
  T row[kMaxRitz];
#pragma unroll
  for (int j = 0; j < kMaxRitz; ++j) {
    if (j < l) {
      T t = X[a * l + j];
#pragma unroll
      for (int k = 0; k < j; ++k) t -= row[k] * Rt[k][j];
      row[j] = t * rinv[j];
    } else {
      row[j] = T(0);
    }
  }
#pragma unroll
  for (int j = 0; j < kMaxRitz; ++j)
    if (j < l) Y[a * l + j] = row[j];
}

// The same for the FP64 path.  Every block factors G redundantly in float-float arithmetic
// (right-looking, one barrier per column, one thread per entry) and applies the same elimination to the identity,
// which leaves W = R^-T; then one thread per entry of X_dst takes its dot
// product with a column of R^-1.  (One thread per row solved the triangular
// system as a chain of l^2 / 2 dependent steps: 29 us a call at 60 rows and 37 us
// at 1024.)  A non-positive pivot
// zeroes that column (rank loss) and flags kStatEigFail.
constexpr int kOrthThreads = kMaxRitz * kMaxRitz;   // one thread per entry of G and W
// Entries of X_dst per block (a multiple of 128): few enough that all SMs share
// the dot products, whose FP64 instructions hold an SM's pipe for 16 clocks a warp
// (1024 entries: 20 us a launch at 60 to 100 rows, 14 us now); every block repeats
// the factorization.
static int orth_entries(int64_t total) {
  constexpr int kSms = 152;   // of a GB300; any other count only changes the split
  return (int)std::min<int64_t>(std::max<int64_t>((total / kSms + 127) / 128 * 128, 128), kOrthThreads);
}
__global__ void __launch_bounds__(kOrthThreads) k_ritz_orth64(const ProblemDev* tab, int src, int entries) {
  const ProblemDev& pr = tab[blockIdx.y];
  const int l = pr.l;
  const int64_t e0 = (int64_t)blockIdx.x * entries, total = pr.d * l;
  if (l <= 0 || e0 >= total) return;
  __shared__ FF G[kMaxRitz][kMaxRitz + 1];   // upper triangle
  __shared__ FF W[kMaxRitz][kMaxRitz + 1];   // lower triangle: R^-T
  __shared__ double Ri[kMaxRitz][kMaxRitz + 1];   // R^-1, upper triangle
  __shared__ float s_tiny;
  const int t = threadIdx.x;
  const int i = t / kMaxRitz, c = t % kMaxRitz;
  const bool mine = i < l && c < l;
  if (mine) {
    if (i <= c) G[i][c] = ff_from(pr.Gm[i * l + c]);
    W[i][c] = FF{i == c ? 1.f : 0.f, 0.f};
  }
  if (t < 32) {
    float tr = t < l ? (float)pr.Gm[t * (l + 1)] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
    if (t == 0) s_tiny = 1e-28f * (tr > 0.f ? tr : 1.f);
  }
  __syncthreads();
  const float tiny = s_tiny;
  for (int j = 0; j < l; ++j) {
    // eliminate below the pivot, row i > j: G[i][c] -= f G[j][c] (c >= i) and
    // W[i][c] -= f W[j][c] (c <= j) with f = G[j][i] / G[j][j]
    const FF gjj = G[j][j];
    const bool ok = gjj.h > tiny;
    if (t == 0 && !ok && blockIdx.x == 0) atomicOr(&pr.status[0], kStatEigFail);
    if (mine && i > j && ok && (c <= j || c >= i)) {
      const FF f = ff_div(G[j][i], gjj);
      if (c <= j) W[i][c] = ff_sub(W[i][c], ff_mul(f, W[j][c]));
      else G[i][c] = ff_sub(G[i][c], ff_mul(f, G[j][c]));
    }
    __syncthreads();
  }
  // R^-1[i][c] = W[c][i] / sqrt(G[c][c]), i <= c
  if (mine) {
    const FF gcc = G[c][c];
    const FF v = gcc.h > tiny && i <= c ? ff_mul(W[c][i], ff_rsqrt(gcc)) : FF{0.f, 0.f};
    Ri[i][c] = (double)v.h + (double)v.l;
  }
  __syncthreads();
  const double* X = ritz_buf<double>(pr, src);
  double* Y = ritz_buf<double>(pr, 1 - src);
  const int64_t e = e0 + t;
  if (t < entries && e < total) {
    const int64_t a = e / l;
    const int j = (int)(e - a * l);
    double s0 = 0.0, s1 = 0.0;   // two chains
    int u = 0;
    for (; u + 1 <= j; u += 2) {
      s0 += X[a * l + u] * Ri[u][j];
      s1 += X[a * l + u + 1] * Ri[u + 1][j];
    }
    if (u <= j) s0 += X[a * l + u] * Ri[u][j];
    Y[e] = s0 + s1;
  }
}

// One-sided (Hestenes) cyclic Jacobi in FP32, one warp per column pair of a
// round (lane i holds row i): U = B and V = I on entry; each round rotates its
// pairs so that their columns of U become orthogonal.  At convergence
// B V = U with orthogonal columns, so the columns of V are eigenvectors and
// lambda_c = v_c . u_c (sign kept).  Squared column norms are carried through
// the rotations (alpha' = alpha - t g, beta' = beta + t g) and recomputed once
// per sweep.  Called by all threads of the block.
struct JacobiPairs {
  float U[kMaxRitz][kMaxRitz + 1], V[kMaxRitz][kMaxRitz + 1];
  float nrm[kMaxRitz];
  float scale;
  int8_t pair_p[kMaxRitz][kMaxRitz / 2], pair_q[kMaxRitz][kMaxRitz / 2];
};
__device__ void jacobi_pairs(JacobiPairs& jp, int l, int sweeps) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int m = (l + 1) & ~1, npairs = m / 2;
  // round-robin schedule (circle method): slot 0 fixed, slot s > 0 holds
  // ((s - 1 + round) mod (m - 1)) + 1; pair w of a round joins slots w and m - 1 - w
  for (int e = tid; e < (m - 1) * npairs; e += blockDim.x) {
    const int round = e / npairs, w = e % npairs;
    const int s1 = w, s2 = m - 1 - w;
    int p = s1 == 0 ? 0 : ((s1 - 1 + round) % (m - 1)) + 1;
    int q = ((s2 - 1 + round) % (m - 1)) + 1;
    if (p > q) { const int x = p; p = q; q = x; }
    jp.pair_p[round][w] = (int8_t)p;
    jp.pair_q[round][w] = (int8_t)q;
  }
  __syncthreads();
  auto refresh_norms = [&]() {
    for (int c = warp; c < l; c += nw) {
      const float u = lane < l ? jp.U[lane][c] : 0.f;
      float a = u * u;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      if (lane == 0) jp.nrm[c] = a;
    }
  };
  refresh_norms();
  __syncthreads();
  if (tid == 0) {
    float mx = 0.f;
    for (int c = 0; c < l; ++c) mx = fmaxf(mx, jp.nrm[c]);
    jp.scale = mx;
  }
  __syncthreads();
  // a pair stays unconverged while the cosine of its columns exceeds 1e-5 and
  // |u_p . u_q| exceeds 2e-6 of the largest squared column norm (below that it
  // is FP32 rounding noise of the small columns)
  const float gabs = 2e-6f * jp.scale;
  // cyclic Jacobi is quadratically convergent; a round costs a few hundred
  // cycles of dependent latency, so the sweep count is the cost (FP32 path: four,
  // the Ritz pairs only shape the preconditioner)
  for (int sweep = 0; sweep < sweeps; ++sweep) {
    int busy = 0;
    for (int round = 0; round < m - 1; ++round) {
      for (int w = warp; w < npairs; w += nw) {
        const int p = jp.pair_p[round][w], q = jp.pair_q[round][w];
        if (q >= l) continue;
        const float up = lane < l ? jp.U[lane][p] : 0.f, uq = lane < l ? jp.U[lane][q] : 0.f;
        float g = up * uq;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        const float al = jp.nrm[p], be = jp.nrm[q];
        if (g == 0.f) continue;
        busy |= fabsf(g) > gabs && fabsf(g) > 1e-5f * sqrtf(al * be);
        // rotation from approximate reciprocals and roots: any orthogonal rotation
        // keeps B V = U exact; these only change how fast the pair converges
        const float zeta = __fdividef(be - al, 2.f * g);
        const float z2 = fmaf(zeta, zeta, 1.f);
        const float tt = copysignf(1.f, zeta) * __fdividef(1.f, fabsf(zeta) + z2 * rsqrtf(z2));
        const float cs = rsqrtf(fmaf(tt, tt, 1.f)), sn = cs * tt;
        if (lane < l) {
          jp.U[lane][p] = cs * up - sn * uq;
          jp.U[lane][q] = sn * up + cs * uq;
          const float vp = jp.V[lane][p], vq = jp.V[lane][q];
          jp.V[lane][p] = cs * vp - sn * vq;
          jp.V[lane][q] = sn * vp + cs * vq;
        }
        if (lane == 0) {
          jp.nrm[p] = fmaxf(al - tt * g, 0.f);
          jp.nrm[q] = fmaxf(be + tt * g, 0.f);
        }
      }
      __syncthreads();
    }
    refresh_norms();
    if (!__syncthreads_or(busy)) break;
  }
  __syncthreads();
}

// The FP32 path's eigenpairs of B = sym(Om^T C Om) (Gm holds Om^T (C Om)): ev
// (descending) and Rm (eigenvectors).
__global__ void k_ritz_jacobi_pairs(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.x];
  const int l = pr.l;
  if (l <= 0) return;
  __shared__ JacobiPairs jp;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  for (int e = tid; e < l * l; e += blockDim.x) {
    const int i = e / l, c = e % l;
    jp.U[i][c] = (float)(0.5 * (pr.Gm[i * l + c] + pr.Gm[c * l + i]));
    jp.V[i][c] = i == c ? 1.f : 0.f;
  }
  jacobi_pairs(jp, l, 4);
  // eigenvalues (Rayleigh quotients) and the descending order
  __shared__ float lam[kMaxRitz];
  for (int c = warp; c < l; c += nw) {
    float a = lane < l ? jp.V[lane][c] * jp.U[lane][c] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) lam[c] = a;
  }
  __syncthreads();
  if (tid < l) {
    const float di = lam[tid];
    int rank = 0;
    for (int u = 0; u < l; ++u) rank += (lam[u] > di) || (lam[u] == di && u < tid);
    pr.ev[rank] = (double)di;
    for (int u = 0; u < l; ++u) pr.Rm[u * l + rank] = (double)jp.V[u][tid];
  }
}


// The FP64 path's eigenpairs of B.  On this GPU an FP64 instruction of a warp
// holds the SM's FP64 pipe for about 16 clocks, so cyclic Jacobi in FP64 (nine
// sweeps of l - 1 rounds) took 486 us at l = 20.  Instead: the FP32 one-sided
// Jacobi above, then two steps of the quadratically convergent refinement of a
// symmetric eigenvector matrix by products (Ogita & Aishima 2018): with
// R = I - X^T X, S = X^T B X and lambda_i = S_ii / (1 - R_ii),
//   X <- X + X E,  E_ij = (S_ij + lambda_j R_ij) / (lambda_j - lambda_i),
// R_ij / 2 where the eigenvalues are too close to separate: 1e-6 -> 1e-12 ->
// rounding where they are separated.  Elsewhere E up to 1e-4 leaves X orthogonal
// to |E|^2 only, so X <- X + X (I - X^T X) / 2 then makes it orthonormal to
// rounding (once or twice): without it the matrix X^T B X that is left has other
// eigenvalues than B (eigenvalues 1 + 1e-5 i, l = 32: wrong in the ninth digit).
// FP64 Jacobi sweeps on (X^T B X, X), one thread per entry and l / 2 disjoint
// rotations per round, finish what is left, if anything (unseparated eigenvalues).
constexpr int kEigThreads = kMaxRitz * kMaxRitz;
__device__ __forceinline__ void jacobi_rotation(double app, double aqq, double apq, double& c, double& s) {
  c = 1.0;
  s = 0.0;
  if (apq != 0.0) {
    const double theta = (aqq - app) / (2.0 * apq);
    const double t = (theta >= 0.0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
    c = 1.0 / sqrt(t * t + 1.0);
    s = t * c;
  }
}

// C = A B or A^T B of l x l matrices, one thread per entry; the caller synchronizes.
template <bool TRANS>
__device__ __forceinline__ void eig_product(const double (*A)[kMaxRitz + 1], const double (*Bm)[kMaxRitz + 1],
                                            double (*Cm)[kMaxRitz + 1], int l) {
  for (int e = threadIdx.x; e < l * l; e += kEigThreads) {
    const int i = e / l, j = e % l;
    double s0 = 0.0, s1 = 0.0;
    int u = 0;
    for (; u + 1 < l; u += 2) {
      s0 += (TRANS ? A[u][i] : A[i][u]) * Bm[u][j];
      s1 += (TRANS ? A[u + 1][i] : A[i][u + 1]) * Bm[u + 1][j];
    }
    if (u < l) s0 += (TRANS ? A[u][i] : A[i][u]) * Bm[u][j];
    Cm[i][j] = s0 + s1;
  }
}

__global__ void __launch_bounds__(kEigThreads) k_ritz_jacobi(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.x];
  const int l = pr.l;
  if (l <= 0) return;
  __shared__ double A[2][kMaxRitz][kMaxRitz + 1];
  __shared__ double V[2][kMaxRitz][kMaxRitz + 1];
  __shared__ union Scratch {
    JacobiPairs jp;                                  // FP32 start
    struct {
      double B[kMaxRitz][kMaxRitz + 1], lam[kMaxRitz];   // refinement (from the end of the FP32 start on)
    } r;
    __device__ Scratch() {}
  } sc;
  __shared__ double cs[kMaxRitz][2];                 // (c, s) of the pair containing index x
  __shared__ int8_t partner[kMaxRitz][kMaxRitz];     // [round][x]
  __shared__ double red_off[kMaxRitz], red_tot[kMaxRitz];
  __shared__ float row_sum[kMaxRitz], row_lam[kMaxRitz];
  __shared__ int go_on;
  const int tid = threadIdx.x;
  const int i = tid / kMaxRitz, j = tid % kMaxRitz;
  const bool mine = i < l && j < l;
  const int m = (l + 1) & ~1;   // even count; index l is a dummy when l is odd
  const double bij = mine ? 0.5 * (pr.Gm[i * l + j] + pr.Gm[j * l + i]) : 0.0;
  if (mine) {
    sc.jp.U[i][j] = (float)bij;
    sc.jp.V[i][j] = i == j ? 1.f : 0.f;
  }
  // circle method: position 0 fixed, the others rotate by one per round
  if (i < m - 1 && j < m) {
    const int round = i, x = j;
    const int pos = x == 0 ? 0 : ((x - 1 - round) % (m - 1) + (m - 1)) % (m - 1) + 1;
    const int ppos = m - 1 - pos;
    partner[round][x] = (int8_t)(ppos == 0 ? 0 : ((ppos - 1 + round) % (m - 1)) + 1);
  }
  __syncthreads();
  jacobi_pairs(sc.jp, l, 8);
  if (mine) V[0][i][j] = (double)sc.jp.V[i][j];
  __syncthreads();
  if (mine) sc.r.B[i][j] = bij;
  __syncthreads();
  // two refinement steps; X in V[0], scratch V[1], A[0], A[1]
  bool usable = true;
  for (int step = 0; step < 2; ++step) {
    eig_product<false>(sc.r.B, V[0], A[0], l);          // B X
    eig_product<true>(V[0], V[0], A[1], l);             // X^T X
    __syncthreads();
    eig_product<true>(V[0], A[0], V[1], l);             // S = X^T B X
    __syncthreads();
    if (tid < l) sc.r.lam[tid] = V[1][tid][tid] / A[1][tid][tid];
    __syncthreads();
    // the separation below which a pair is left alone: twice the largest row
    // sum of |S - Lambda| + |Lambda| |R| (FP32 will do for it)
    const double r = mine ? (i == j ? 1.0 : 0.0) - A[1][i][j] : 0.0;
    if (i < l) {
      const float li = fabsf((float)sc.r.lam[i]);
      float v = mine ? fabsf((float)(V[1][i][j] - (i == j ? sc.r.lam[i] : 0.0))) + li * fabsf((float)r) : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (j == 0) {
        row_sum[i] = v < INFINITY ? v : INFINITY;   // NaN as infinity: the maximum below would drop it
        row_lam[i] = li;
      }
    }
    __syncthreads();
    float delta = 0.f, lmax = 0.f;
    for (int u = 0; u < l; ++u) {
      delta = fmaxf(delta, row_sum[u]);
      lmax = fmaxf(lmax, row_lam[u]);
    }
    delta *= 2.f;
    // a start that is no near eigenbasis (values beyond FP32's range, say):
    // FP64 Jacobi from the beginning
    if (step == 0 && !(delta <= 1e-2f * lmax && delta < INFINITY)) {
      usable = false;
      break;
    }
    if (mine) {
      // E to FP32's relative accuracy: it is the size of the error that this step
      // removes.  Entries above 1e-4 (close eigenvalues) would cost orthogonality
      // in second order and are left to the sweeps below.
      const float gap = (float)(sc.r.lam[j] - sc.r.lam[i]);
      const float e = (float)(V[1][i][j] + sc.r.lam[j] * r) / gap;
      A[0][i][j] = i != j && fabsf(gap) > delta && fabsf(e) < 1e-4f ? (double)e : 0.5 * r;
    }
    __syncthreads();
    eig_product<false>(V[0], A[0], V[1], l);            // X E
    __syncthreads();
    if (mine) V[0][i][j] += V[1][i][j];
    __syncthreads();
  }
  // X orthonormal to rounding: a step squares the error (3/4 R^2), so from 1e-9 one is enough
  for (int step = 0; usable && step < 3; ++step) {
    eig_product<true>(V[0], V[0], A[1], l);             // X^T X
    __syncthreads();
    const double r = mine ? (i == j ? 1.0 : 0.0) - A[1][i][j] : 0.0;
    if (mine) A[0][i][j] = 0.5 * r;
    if (!__syncthreads_or(fabs(r) > 1e-15)) break;
    eig_product<false>(V[0], A[0], V[1], l);
    const int again = __syncthreads_or(fabs(r) > 1e-9);
    if (mine) V[0][i][j] += V[1][i][j];
    __syncthreads();
    if (!again) break;
  }
  if (usable) {
    eig_product<false>(sc.r.B, V[0], A[1], l);
    __syncthreads();
    eig_product<true>(V[0], A[1], A[0], l);             // X^T B X
  } else if (mine) {
    A[0][i][j] = bij;
    V[0][i][j] = i == j ? 1.0 : 0.0;
  }
  int cur = 0;
  __syncthreads();
  // off-diagonal norm within 1e-15 of the whole: done, usually before the first sweep
  const int max_sweeps = 30;
  const double eps = 1e-30;
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    {
      // off-diagonal and total squared norms: warp i holds row i
      double v = mine ? A[cur][i][j] * A[cur][i][j] : 0.0;
      double o = (mine && i != j) ? v : 0.0;
#pragma unroll
      for (int sh = 16; sh > 0; sh >>= 1) {
        v += __shfl_xor_sync(0xffffffffu, v, sh);
        o += __shfl_xor_sync(0xffffffffu, o, sh);
      }
      if (j == 0) { red_tot[i] = v; red_off[i] = o; }
      __syncthreads();
      if (tid < 32) {
        double to = red_tot[tid], of = red_off[tid];
#pragma unroll
        for (int sh = 16; sh > 0; sh >>= 1) {
          to += __shfl_xor_sync(0xffffffffu, to, sh);
          of += __shfl_xor_sync(0xffffffffu, of, sh);
        }
        if (tid == 0) go_on = of > eps * to;
      }
      __syncthreads();
    }
    if (!go_on) break;
    for (int round = 0; round < m - 1; ++round) {
      if (tid < l) {
        const int x = tid, y = partner[round][x];
        if (x < y && y < l) {
          double c, s;
          jacobi_rotation(A[cur][x][x], A[cur][y][y], A[cur][x][y], c, s);
          cs[x][0] = c; cs[x][1] = s;
          cs[y][0] = c; cs[y][1] = s;
        } else if (y >= l) {
          cs[x][0] = 1.0; cs[x][1] = 0.0;
        }
      }
      __syncthreads();
      if (mine) {
        // coefficients of row/column index u: new_u = al * X_p + be * X_q for its pair (p < q)
        auto coef = [&](int u, int& p, int& q, double& al, double& be) {
          const int v2 = partner[round][u];
          if (v2 >= l) { p = u; q = u; al = 1.0; be = 0.0; return; }
          const double c = cs[u][0], s = cs[u][1];
          if (u < v2) { p = u; q = v2; al = c; be = -s; }
          else { p = v2; q = u; al = s; be = c; }
        };
        int pi, qi, pj, qj;
        double ai, bi, aj, bj;
        coef(i, pi, qi, ai, bi);
        coef(j, pj, qj, aj, bj);
        const double (*Ac)[kMaxRitz + 1] = A[cur];
        double nv;
        if (pi == qi && pj == qj) nv = Ac[i][j];
        else if (pi == qi) nv = aj * Ac[i][pj] + bj * Ac[i][qj];
        else if (pj == qj) nv = ai * Ac[pi][j] + bi * Ac[qi][j];
        else nv = ai * (aj * Ac[pi][pj] + bj * Ac[pi][qj]) + bi * (aj * Ac[qi][pj] + bj * Ac[qi][qj]);
        A[1 - cur][i][j] = nv;
        V[1 - cur][i][j] = pj == qj ? V[cur][i][j] : aj * V[cur][i][pj] + bj * V[cur][i][qj];
      }
      __syncthreads();
      cur = 1 - cur;
    }
  }
  // descending order: rank of each diagonal entry
  if (tid < l) {
    const double di = A[cur][tid][tid];
    int rank = 0;
    for (int u = 0; u < l; ++u) {
      const double du = A[cur][u][u];
      rank += (du > di) || (du == di && u < tid);
    }
    pr.ev[rank] = di;
    for (int u = 0; u < l; ++u) pr.Rm[u * l + rank] = V[cur][u][tid];
  }
}

// Phi = basis V_k, C Phi = image V_k (stored in T), theta = top k eigenvalues;
// one thread per entry of both (a thread per row ran 2 l k dependent steps on a
// couple of SMs: 25 us in FP64 at 60 rows, 50 us at 1024).
constexpr int kVecEntries = 128;
template <typename T>
__global__ void __launch_bounds__(kVecEntries) k_ritz_vectors(const ProblemDev* tab, int basis) {
  const ProblemDev& pr = tab[blockIdx.y];
  const int l = pr.l, k = pr.kR;
  const int64_t e0 = (int64_t)blockIdx.x * kVecEntries, total = pr.d * k;
  if (k <= 0 || e0 >= total) return;
  __shared__ T Vk[kMaxRitz][kMaxK];
  for (int e = threadIdx.x; e < l * k; e += kVecEntries) Vk[e / k][e % k] = to_t<T>(pr.Rm[(e / k) * l + e % k]);
  __syncthreads();
  const int64_t e = e0 + threadIdx.x;
  if (e < total) {
    const int64_t a = e / k;
    const int j = (int)(e - a * k);
    const T* q = ritz_buf<T>(pr, basis) + a * l;
    const T* c = ritz_buf<T>(pr, 1 - basis) + a * l;
    T ph = T(0), cp = T(0);
#pragma unroll 4
    for (int i = 0; i < l; ++i) {
      ph += q[i] * Vk[i][j];
      cp += c[i] * Vk[i][j];
    }
    tp<T>(pr.Phi)[e] = ph;
    tp<T>(pr.CPhi)[e] = cp;
    if (a == 0) pr.theta[j] = pr.ev[j];
  }
}

// Gram matrices of the stored Phi and A = C Phi in FP64:
// gram[0] = Phi^T Phi, gram[1] = A^T Phi, gram[2] = A^T A.  One block per entry.
template <typename T>
__global__ void k_ritz_grams(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.y];
  const int k = pr.kR;
  const int e = blockIdx.x;
  if (k <= 0 || e >= 3 * k * k) return;
  const int which = e / (k * k), i = (e / k) % k, j = e % k;
  const T* Phi = tp<const T>(pr.Phi);
  const T* A = tp<const T>(pr.CPhi);
  const T* L = which == 0 ? Phi : A;
  const T* Rr = which == 2 ? A : Phi;
  DotAcc<T> acc;
  for (int64_t a = threadIdx.x; a < pr.d; a += blockDim.x) acc.add_prod(L[a * k + i], Rr[a * k + j]);
  DotAcc<T> accs[1] = {acc};
  double out[1];
  __shared__ double scratch[2 * kThreads / 32];
  block_sum<1>(accs, out, scratch);
  if (threadIdx.x == 0) pr.gram[e] = out[0];
}

// tile = true: the BF16 block-tile path, whose C exists only as stored blocks;
// the matvec of the range finder then runs over those blocks (FP32 basis).
template <typename T>
static void launch_ritz_t(const ProblemTable& tab, const ProblemDev* dtab, cudaStream_t st, bool tile = false) {
  int64_t dl = 0, dmax = 0;
  int lmax = 0, kmax = 0;
  for (int i = 0; i < tab.count; ++i) {
    const ProblemDev& p = tab.p[i];
    dl = p.d * p.l > dl ? p.d * p.l : dl;
    dmax = p.d > dmax ? p.d : dmax;
    lmax = p.l > lmax ? p.l : lmax;
    kmax = p.kR > kmax ? p.kR : kmax;
  }
  if (lmax <= 0 || kmax <= 0) return;
  const dim3 gdl((unsigned)((dl + 255) / 256), tab.count);
  const dim3 gd((unsigned)((dmax + 255) / 256), tab.count);
  const int oe = orth_entries(dl * tab.count);
  const dim3 go((unsigned)((dl + oe - 1) / oe), tab.count);
  const dim3 gv((unsigned)((dmax * kmax + kVecEntries - 1) / kVecEntries), tab.count);
  const dim3 gdw((unsigned)((dmax * 32 + 255) / 256), tab.count);   // one warp per row
  const dim3 gll((unsigned)(lmax * lmax), tab.count);
  int cur = 0;   // buffer holding the current basis candidate
  auto matvec = [&]() {   // buf[1 - cur] = C buf[cur]
    if (tile) {
      launch_tile_ritz_matvec(tab, dtab, cur, st);
      return;
    }
    k_ritz_matvec<T><<<gdw, 256, 0, st>>>(dtab, cur);
    note_launches(1);
  };
  auto orth = [&](int x) {
    if constexpr (sizeof(T) == 8) k_ritz_orth64<<<go, kOrthThreads, 0, st>>>(dtab, x, oe);
    else k_ritz_orth<T><<<gd, 256, 0, st>>>(dtab, x);
  };
  auto orth2 = [&](int x) {   // orthonormalize buf[x] in place (scratch: the other buffer)
    k_ritz_gram<T><<<gll, 256, 0, st>>>(dtab, x, x, 1);
    orth(x);                                              // buf[1-x] = buf[x] R^-1
    k_ritz_gram<T><<<gll, 256, 0, st>>>(dtab, 1 - x, 1 - x, 1);
    orth(1 - x);                                          // buf[x] = buf[1-x] R^-1
    note_launches(4);
  };
  k_ritz_omega<T><<<gdl, 256, 0, st>>>(dtab);               // buf0 = Omega
  note_launches(1);
  matvec();                                                 // buf1 = C buf0
  cur = 1;
  for (int it = 0; it < tab.p[0].power_iters; ++it) {
    orth2(cur);                                             // buf[cur] orthonormal
    matvec();                                               // buf[1-cur] = C buf[cur]
    cur = 1 - cur;
  }
  orth2(cur);                                               // basis in buf[cur]
  matvec();                                                 // image in buf[1-cur]
  k_ritz_gram<T><<<gll, 256, 0, st>>>(dtab, cur, 1 - cur, 0);   // Gm = Q^T (C Q)
  if (sizeof(T) == 4) k_ritz_jacobi_pairs<<<tab.count, 32 * ((lmax + 1) / 2), 0, st>>>(dtab);
  else k_ritz_jacobi<<<tab.count, kEigThreads, 0, st>>>(dtab);
  k_ritz_vectors<T><<<gv, kVecEntries, 0, st>>>(dtab, cur);
  k_ritz_grams<T><<<dim3(3 * kmax * kmax, tab.count), 256, 0, st>>>(dtab);
  note_launches(4);
  if (!tile) launch_pcg_phit(tab, dtab, st);
}

void launch_ritz(const ProblemTable& tab, const ProblemDev* dtab, cudaStream_t st) {
  if (tab.p[0].precision == 0) {
    launch_ritz_t<double>(tab, dtab, st);
    return;
  }
  if (tab.p[0].precision == 2) {
    launch_ritz_t<float>(tab, dtab, st, true);
    return;
  }
  // FP32: one cluster launch for the whole stage when every problem fits it
  bool fused = true;
  for (int i = 0; i < tab.count; ++i) {
    const ProblemDev& p = tab.p[i];
    fused &= p.l > 0 && p.kR > 0 && p.l <= kMaxRitz && p.kR <= kMaxK && ritz_cluster_fits(p.d, p.l);
  }
  if (fused && launch_ritz_cluster(tab, dtab, st) == 0) return;
  launch_ritz_t<float>(tab, dtab, st);
}

}  // namespace infoesrf
