// a6-a8, BF16 path: batched shifted PCG over every (node, member) system and
// the mean system (App. E, Eq. normalized_linear_solve; Golub & Van Loan
// Alg. 11.5.1) with the limited-memory preconditioner of App. E, as a
// sequence of kernels per iteration over all systems at once:
//
//   1. y_j = sigma_j p_j + C p_j and row-tile partials of p_j^T y_j
//      (tensor-core block-tile matvec, tile_matvec.cu);
//   2. alpha_j = rho_j / p_j^T y_j (FP64, partials summed in a fixed order);
//   3. x_j += alpha_j p_j, r_j -= alpha_j y_j, and partials of r^T r,
//      f = Phi^T r, g = (C Phi)^T r (FP32 over 512 rows, FP64 across row blocks);
//   4. per system: convergence test ||r|| <= tol ||b||, the preconditioner
//      coefficients t = T^-1 f, c = (beta_lmp - sigma) t - T^-1 (g + sigma f - G_q t)
//      with G_q = (C_q Phi)^T (C_q Phi), rho' = r^T z = r^T r - g.t + f.c and
//      beta = rho' / rho (FP64);
//   5. p_j = bf16(z_j + beta_j p_j), z = r - (C Phi) t + Phi c.
//
// Learned correction (2-D observation lattices with a model; tile_learn.cu):
// after step 3, u = S r and u^T u; step 4 takes rho = a (r^T P^-1 r) + u^T u,
// step 5 z = a P^-1 r + S u.  A learned system that breaks down or reaches
// the iteration cap is solved again from the start without the term (plain
// PCG as the fallback), after the other systems.
//
// The directions are stored in BF16 and the same BF16 vector enters the
// matvec and the update of x (step 3), so x and r stay consistent:
// r = b - C_q x up to the accuracy of the product (C kept as hi + lo BF16
// planes, about 16 significant bits; products exact, FP32 accumulation).
// Rounding p only perturbs the conjugacy of the directions, not the system
// that is solved.  Converged systems leave the lists of running systems, and with them
// the matvec.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "info_esrf.h"
#include "internal.h"
#include "tile_mma.cuh"

namespace infoesrf {

namespace {

constexpr int kDotRows = kTileDotRows;   // rows per CTA of the update (and per partial dot product)
constexpr int kVecWarps = 4;       // row chunks per CTA of the direction kernel, one per warp
constexpr int kVecThreads = 32 * kVecWarps;
constexpr int kMaxGroup = 32;      // systems per CTA of the direction kernel at most
// per-system FP64 scalars in sysd[j][8]
enum { kRho = 0, kBn2 = 1, kRr = 2, kFirst = 3 };

__device__ __forceinline__ double sys_sigma(const ProblemDev& pr, int64_t j) {
  if (j < pr.mean_sys) return 1.0;
  const int64_t q = (j - pr.mean_sys) / pr.N;
  return pr.s[q] + 1.0;
}

// x = 0, r = b and the per-system state (mode 0), or (mode 1) the
// per-system state of the systems marked for a retry without the learned
// term, whose vectors k_tpcg_retry_vectors has reset.
__global__ void k_tpcg_init(const ProblemDev* dpr, int mode, int allow_learn) {
  const ProblemDev& pr = *dpr;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t J = pr.nsys;
  if (i < J && (mode == 0 || pr.learn_on[i] == 2)) {
    double* sd = pr.sysd + i * 8;
    sd[kRho] = 0.0;
    sd[kBn2] = 0.0;
    sd[kRr] = 0.0;
    sd[kFirst] = 1.0;
    pr.sigmaf[i] = (float)sys_sigma(pr, i);
    pr.active[i] = 1;
    pr.iters[i] = 0;
    pr.relres[i] = 0.0;
    if (pr.learn_on) {
      int on = 0;
      if (mode == 0 && allow_learn && pr.learned_model && pr.lat_info[0] == 1) {
        const int64_t q = i < pr.mean_sys ? pr.Q : (i - pr.mean_sys) / pr.N;
        on = pr.learn_coef[q * kLearnOut] > 0.f ? 1 : 0;
        if (on) atomicAdd(&pr.lat_info[8], 1);
      }
      pr.learn_on[i] = on;
    }
  }
  if (i == 0)
    for (int c = 0; c < 4; ++c) pr.nactive[c] = 0;
  if (mode != 0 || i >= J * pr.d_pad) return;
  const int64_t j = i / pr.d_pad, a = i % pr.d_pad;
  float b = 0.f;
  const int32_t src = a < pr.d ? pr.tpos_src[a] : -1;
  if (src >= 0) {
    if (j < pr.mean_sys) b = (float)pr.bmean[src];
    else b = pr.Wp[a * pr.N + (j - pr.mean_sys) % pr.N] * pr.rinvp[a];
  }
  pr.Xv[i] = 0.f;
  pr.Rv[i] = b;
}

// x = 0, r = b for the systems marked for a retry (learn_on == 2).
__global__ void k_tpcg_retry_vectors(const ProblemDev* dpr) {
  const ProblemDev& pr = *dpr;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= pr.nsys * pr.d_pad) return;
  const int64_t j = i / pr.d_pad, a = i % pr.d_pad;
  if (pr.learn_on[j] != 2) return;
  float b = 0.f;
  const int32_t src = a < pr.d ? pr.tpos_src[a] : -1;
  if (src >= 0) {
    if (j < pr.mean_sys) b = (float)pr.bmean[src];
    else b = pr.Wp[a * pr.N + (j - pr.mean_sys) % pr.N] * pr.rinvp[a];
  }
  pr.Xv[i] = 0.f;
  pr.Rv[i] = b;
}

// A learned system that failed: stop it and mark it for the retry.
__device__ __forceinline__ void mark_retry(const ProblemDev& pr, int64_t j) {
  pr.active[j] = 0;
  pr.learn_on[j] = 2;
  atomicAdd(&pr.lat_info[7], 1);
}

// Systems are addressed in two ways.  X, R and the FP64 scalars belong to the
// system j.  What one iteration hands to the next kernel (the directions P,
// their images Y, the partial sums and the coefficients) is kept by position
// in the iteration's list of running systems: list[pos] = j, and the next
// list's src[pos] = position in the list before.  So the matvec runs over
// consecutive rows of P (one TMA box per stage, no idle columns), and a kernel
// finds what it needs one load after the list.  The lists are appended with
// atomics: their order differs from run to run, which no result depends on
// (every column of the product and every sum belongs to one system).
//
// Counts rotate over three slots: iteration `it` runs cnt[it % 3] systems,
// appends the survivors to cnt[(it + 1) % 3] and clears cnt[(it + 2) % 3].
__device__ __forceinline__ int64_t list_count(const ProblemDev& pr, const int32_t* list, int it) {
  return list ? pr.nactive[it % 3] : pr.nsys;
}

// alpha = rho_j / p^T y of the system at position pos by one warp (lanes over
// the row-tile partials, a fixed shuffle tree; every lane returns it).
// record: this warp also keeps the iteration count and handles a breakdown
// (p^T y <= 0 or not finite), which stops the system with alpha = 0.
__device__ __forceinline__ double warp_alpha(const ProblemDev& pr, int64_t j, int64_t pos, int it, bool record,
                                             int lane) {
  double pap = 0.0;
  const float* src = pr.pty + pos * pr.nrt;
  const double rho = pr.sysd[j * 8 + kRho];
  for (int64_t t = lane; t < pr.nrt; t += 32) pap += (double)src[t];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pap += __shfl_xor_sync(0xffffffffu, pap, o);
  const bool ok = pap > 0.0 && isfinite(pap);
  const double al = ok ? rho / pap : 0.0;
  if (record && lane == 0) {
    if (ok) {
      pr.iters[j] = it;
    } else if (pr.learn_on && pr.learn_on[j] == 1) {
      mark_retry(pr, j);
    } else {
      pr.active[j] = 0;
      atomicOr(&pr.status[0], kStatBreakdown);
    }
  }
  return al;
}

// Step 2 for problems of many row tiles: one warp per position.  With few row
// tiles (kFusedAlpha) the update kernel forms alpha itself.
__global__ void k_tpcg_alpha(const ProblemDev* dpr, int it, const int32_t* list) {
  const ProblemDev& pr = *dpr;
  const int64_t pos = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (pos >= list_count(pr, list, it)) return;
  const double al = warp_alpha(pr, list[pos], pos, it, true, lane);
  if (lane == 0) pr.alphaf[pos] = (float)al;
}
// Row tiles up to which the update kernel sums p^T y itself: every one of its
// CTAs repeats the sum for its systems, nrt / 32 FP64 additions a lane.  At 32
// row tiles a separate launch cost 4.3 us of a 110 us iteration; at 512 the
// repeats would read 30 MB of partials per iteration.
constexpr int kFusedAlpha = 128;

// [Phi | C Phi] transposed, phiT[m][a] (m < k: Phi, then C Phi; zero at the
// padding rows): the vector kernels read a column at four consecutive rows
// with one coalesced 16-byte load.  Built once per analysis.
__global__ void k_tpcg_phit(const ProblemDev* dpr) {
  const ProblemDev& pr = *dpr;
  const int k = pr.kR;
  const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= pr.d_pad) return;
  const float* P = reinterpret_cast<const float*>(pr.Phi);
  const float* A = reinterpret_cast<const float*>(pr.CPhi);
  const bool in = a < pr.d;
  float* out = reinterpret_cast<float*>(pr.phiT);
  for (int m = 0; m < k; ++m) {
    out[(int64_t)m * pr.d_pad + a] = in ? P[a * k + m] : 0.f;
    out[(int64_t)(k + m) * pr.d_pad + a] = in ? A[a * k + m] : 0.f;
  }
}

__device__ __forceinline__ float4 bf16x4(uint2 w) {
  return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                     __uint_as_float(w.y & 0xffff0000u));
}

// Step 3 (update = 1 or 2: x += alpha p, r -= alpha y first; 2 forms alpha
// here) and the partial dot products r^T r, Phi^T r, (C Phi)^T r over the
// CTA's kDotRows rows, dots[j][block][NVD].
//
// Sixteen lanes serve the rows of a system, four consecutive rows per lane and
// step; a thread carries SPT systems side by side, so one 16-byte read of a
// staged column serves 4 SPT FMAs.  The columns come as 2 k bulk copies of the
// transposed [Phi | C Phi] on one mbarrier, under which the first vectors
// load; the next step's vectors load under the current step's FMAs.  HBM-bound
// at large sizes (22 bytes a row and system), latency-bound at small ones.
// (A transposing stage by all threads and one system per thread took 13.2 us a
// launch at 4096 rows x 66 systems on average and 67 us at 65,536 x 145.)
// The order of every sum is that of one thread per (system, lane) with rows
// ascending, whatever SPT.
constexpr int kRowLanes = 16;
constexpr int kUpdThreads = 128;
constexpr int kUpdSlots = kUpdThreads / kRowLanes;   // 8

struct VecStep {
  float4 r, y, x;
  uint2 p;
};

template <int NV32, int SPT>
__global__ void __launch_bounds__(kUpdThreads) k_tpcg_update(const ProblemDev* dpr, int update, const int32_t* list,
                                                             const __nv_bfloat16* P, int it) {
  grid_dependency_wait();
  constexpr int kSys = kUpdSlots * SPT;
  extern __shared__ float4 phs_dyn4[];   // [2 k][kDotRows / 4]
  __shared__ alignas(8) uint64_t bar;
  __shared__ int32_t sys[kSys];
  __shared__ float als[kSys];
  const ProblemDev& pr = *dpr;
  const int k = pr.kR, NVD = tile_dot_values(k);
  const int64_t dp = pr.d_pad;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t count = list_count(pr, list, it);
  const int64_t group = (int64_t)blockIdx.z * gridDim.y + blockIdx.y;
  if (blockIdx.x == 0 && group == 0 && threadIdx.x == 0) pr.nactive[(it + 2) % 3] = 0;
  const int64_t g0 = group * kSys;
  if (g0 >= count) return;
  const int64_t abase = (int64_t)blockIdx.x * kDotRows;
  const int nrow = (int)(dp - abase < kDotRows ? dp - abase : kDotRows);   // a multiple of 128
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
    if (k > 0) mbar_arrive_expect_tx(&bar, (uint32_t)(2 * k * nrow * 4));
    for (int m = 0; m < 2 * k; ++m)
      bulk_load(phs_dyn4 + m * (kDotRows / 4), reinterpret_cast<const float*>(pr.phiT) + (int64_t)m * dp + abase, (uint32_t)(nrow * 4), &bar);
  }
  if (threadIdx.x < kSys) {
    const int64_t pos = g0 + threadIdx.x;
    const int64_t j = pos < count ? (list ? list[pos] : pos) : -1;
    als[threadIdx.x] = j >= 0 && update == 1 ? pr.alphaf[pos] : 0.f;
    sys[threadIdx.x] = j >= 0 && (list || pr.active[j]) ? (int32_t)j : -1;
  }
  __syncthreads();
  const int slot = threadIdx.x / kRowLanes, r0 = threadIdx.x % kRowLanes;
  int64_t base[SPT], pbase[SPT];   // first element of each of the thread's systems (X, R) and positions (Y, P)
#pragma unroll
  for (int u = 0; u < SPT; ++u) {
    const int s = slot * SPT + u;
    base[u] = sys[s] < 0 ? -1 : (int64_t)sys[s] * dp + abase;
    pbase[u] = (g0 + s) * dp + abase;
  }
  float acc[SPT][32 * NV32];
#pragma unroll
  for (int u = 0; u < SPT; ++u)
#pragma unroll
    for (int v = 0; v < 32 * NV32; ++v) acc[u][v] = 0.f;
  VecStep cur[SPT], nxt[SPT];
  auto load = [&](VecStep (&w)[SPT], int r4) {
#pragma unroll
    for (int u = 0; u < SPT; ++u) {
      w[u].r = make_float4(0.f, 0.f, 0.f, 0.f);
      if (base[u] < 0 || r4 >= nrow) continue;
      w[u].r = *reinterpret_cast<const float4*>(pr.Rv + base[u] + r4);
      if (update) {
        w[u].y = *reinterpret_cast<const float4*>(pr.Yv + pbase[u] + r4);
        w[u].x = *reinterpret_cast<const float4*>(pr.Xv + base[u] + r4);
        w[u].p = *reinterpret_cast<const uint2*>(P + pbase[u] + r4);
      }
    }
  };
  load(cur, 4 * r0);   // in flight while alpha is formed
  if (update == 2) {
    for (int s = warp; s < kSys; s += kUpdThreads / 32) {
      const int j = sys[s];
      if (j < 0) continue;
      const double al = warp_alpha(pr, j, g0 + s, it, blockIdx.x == 0, lane);
      if (lane == 0) als[s] = (float)al;
    }
    __syncthreads();
  }
  float al[SPT];
#pragma unroll
  for (int u = 0; u < SPT; ++u) al[u] = als[slot * SPT + u];
  if (k > 0 && !mbar_wait(&bar, 0)) {
    atomicOr(&pr.status[0], kStatTimeout);
    return;
  }
#pragma unroll 1
  for (int r4 = 4 * r0; r4 < nrow; r4 += 4 * kRowLanes) {
    load(nxt, r4 + 4 * kRowLanes);
#pragma unroll
    for (int u = 0; u < SPT; ++u) {
      if (update && base[u] >= 0) {
        const float4 p = bf16x4(cur[u].p);
        cur[u].x.x = fmaf(al[u], p.x, cur[u].x.x);
        cur[u].x.y = fmaf(al[u], p.y, cur[u].x.y);
        cur[u].x.z = fmaf(al[u], p.z, cur[u].x.z);
        cur[u].x.w = fmaf(al[u], p.w, cur[u].x.w);
        cur[u].r.x = fmaf(-al[u], cur[u].y.x, cur[u].r.x);
        cur[u].r.y = fmaf(-al[u], cur[u].y.y, cur[u].r.y);
        cur[u].r.z = fmaf(-al[u], cur[u].y.z, cur[u].r.z);
        cur[u].r.w = fmaf(-al[u], cur[u].y.w, cur[u].r.w);
        *reinterpret_cast<float4*>(pr.Xv + base[u] + r4) = cur[u].x;
        *reinterpret_cast<float4*>(pr.Rv + base[u] + r4) = cur[u].r;
      }
      acc[u][0] = fmaf(cur[u].r.x, cur[u].r.x, acc[u][0]);
      acc[u][0] = fmaf(cur[u].r.y, cur[u].r.y, acc[u][0]);
      acc[u][0] = fmaf(cur[u].r.z, cur[u].r.z, acc[u][0]);
      acc[u][0] = fmaf(cur[u].r.w, cur[u].r.w, acc[u][0]);
    }
    const float4* col4 = phs_dyn4 + r4 / 4;
#pragma unroll
    for (int m = 0; m < 32 * NV32 - 1; ++m) {
      if (m < 2 * k) {
        const float4 f = col4[m * (kDotRows / 4)];
#pragma unroll
        for (int u = 0; u < SPT; ++u) {
          float t = acc[u][1 + m];
          t = fmaf(f.x, cur[u].r.x, t);
          t = fmaf(f.y, cur[u].r.y, t);
          t = fmaf(f.z, cur[u].r.z, t);
          acc[u][1 + m] = fmaf(f.w, cur[u].r.w, t);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < SPT; ++u) cur[u] = nxt[u];
  }
  // reduce over the 16 row lanes of each system (a half-warp): a reduce-scatter
  // with offsets 8, 4, 2, 1 leaves two values of each 32-value chunk per lane
  const int nsub = gridDim.x;
  const int vlane = 16 * ((r0 >> 3) & 1) + 8 * ((r0 >> 2) & 1) + 4 * ((r0 >> 1) & 1) + 2 * (r0 & 1);
#pragma unroll
  for (int u = 0; u < SPT; ++u) {
#pragma unroll
    for (int c = 0; c < NV32; ++c) {
      float* v = acc[u] + 32 * c;
#pragma unroll
      for (int off = 8, width = 16; off >= 1; off >>= 1, width >>= 1) {
        const bool up = (r0 & off) != 0;
#pragma unroll
        for (int i = 0; i < width; ++i) {
          const float send = up ? v[i] : v[i + width];
          const float keep = up ? v[i + width] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
      }
      float* out = pr.dots + ((g0 + slot * SPT + u) * nsub + blockIdx.x) * NVD;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int vi = 32 * c + vlane + i;
        if (base[u] >= 0 && vi <= 2 * k) out[vi] = v[i];
      }
    }
  }
}

// Step 4: one CTA per position.  The row-chunk partials are summed in FP64
// (warp w takes the chunks w, w + 8, ..., lane v the value v; then the warps in
// order: the same order every call), warp 0 then runs the k x k algebra of the
// preconditioner with one lane per Ritz vector and the k^2 products spread over
// the CTA.  (One thread per system ran k^2 dependent FP64 steps: 42 us a
// launch, a quarter to a third of an iteration on small problems.)
constexpr int kScalThreads = 256;
__global__ void __launch_bounds__(kScalThreads) k_tpcg_scalars(const ProblemDev* dpr, int nsub, int last,
                                                               const int32_t* list, int32_t* next, int32_t* src,
                                                               int it) {
  grid_dependency_wait();
  const ProblemDev& pr = *dpr;
  const int64_t pos = blockIdx.x;
  const int64_t j = pos < list_count(pr, list, it) ? (list ? list[pos] : pos) : -1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (blockIdx.x == 0 && tid == 0) pr.nactive[3] = pr.status[0];   // timeouts and overflow are set by earlier kernels
  if (j < 0 || !pr.active[j]) return;
  const int k = pr.kR, NVD = tile_dot_values(k);
  __shared__ double part[kScalThreads / 32][2 * kMaxK + 2];
  __shared__ double v[2 * kMaxK + 2];   // r^T r, f = Phi^T r, g = (C Phi)^T r, u^T u
  __shared__ double t_s[kMaxK], ti_s[kMaxK];
  __shared__ double gt_s[kMaxK][kMaxK + 1];
  __shared__ int go;
  // everything that does not depend on the sums is loaded before them, so that
  // the launch costs few of the memory's latencies one after another
  const double sigma = sys_sigma(pr, j);
  double* sd = pr.sysd + j * 8;
  const double rho0 = sd[kRho], bn20 = sd[kBn2];
  const bool first = sd[kFirst] != 0.0;
  const bool lrn = pr.learn_on && pr.learn_on[j] == 1;
  float la = 0.f;
  if (lrn) la = pr.learn_coef[(j < pr.mean_sys ? pr.Q : (j - pr.mean_sys) / pr.N) * kLearnOut];
  const double beta0 = pr.scal[1];   // beta_lmp - sigma
  // G_q = A^T A + sigma (A^T Phi + Phi^T A) + sigma^2 Phi^T Phi, entries tid, tid + 256, ..
  constexpr int kGramPer = (kMaxK * kMaxK + kScalThreads - 1) / kScalThreads;
  double G[kGramPer];
#pragma unroll
  for (int i = 0; i < kGramPer; ++i) {
    const int e = tid + i * kScalThreads;
    if (e < k * k)
      G[i] = pr.gram[2 * k * k + e] + sigma * (pr.gram[k * k + e] + pr.gram[k * k + (e % k) * k + e / k]) +
             sigma * sigma * pr.gram[e];
  }
  if (tid < k) ti_s[tid] = 1.0 / (pr.theta[tid] + sigma);
  for (int e = lane; e < NVD; e += 32) {
    double sum = 0.0;
    const float* d = pr.dots + pos * nsub * NVD + e;
#pragma unroll 4
    for (int cb = warp; cb < nsub; cb += kScalThreads / 32) sum += (double)d[(int64_t)cb * NVD];
    part[warp][e] = sum;
  }
  __syncthreads();
  if (tid < NVD) {
    double sum = 0.0;
#pragma unroll
    for (int w = 0; w < kScalThreads / 32; ++w) sum += part[w][tid];
    v[tid] = sum;
    if (tid >= 1 && tid <= k) t_s[tid - 1] = sum * ti_s[tid - 1];
  }
  __syncthreads();
  const double rr = v[0];
  if (tid == 0) {
    go = 0;
    const double bn2 = first ? rr : bn20;
    if (first) sd[kBn2] = rr;
    sd[kRr] = rr;
    pr.relres[j] = bn2 > 0.0 ? sqrt(rr / bn2) : 0.0;
    bool act = true;
    if (pr.fixed_iters <= 0 && !(rr > pr.tol * pr.tol * bn2)) act = false;
    if (!isfinite(rr) && lrn) {
      mark_retry(pr, j);
    } else {
      if (!(rr > 0.0) || !isfinite(rr)) act = false;
      if (last && act) {
        // iteration cap reached with the system still running
        if (lrn && pr.fixed_iters <= 0) {
          mark_retry(pr, j);
        } else {
          if (pr.fixed_iters <= 0) atomicOr(&pr.status[0], kStatNotConverged);
          pr.active[j] = 0;
        }
        act = false;
      } else if (!act) {
        pr.active[j] = 0;
      }
      go = act ? 1 : 0;
    }
  }
  // G_q t, one product per thread
#pragma unroll
  for (int i = 0; i < kGramPer; ++i) {
    const int e = tid + i * kScalThreads;
    if (e < k * k) gt_s[e / k][e % k] = G[i] * t_s[e % k];
  }
  __syncthreads();
  if (!go || warp != 0) return;
  int at = 0;   // the system's position in the next list; needed last
  if (lane == 0) at = atomicAdd(&pr.nactive[(it + 1) % 3], 1);
  float* lc = pr.lcoef + pos * 2 * kMaxK;
  double gt = 0.0, fc = 0.0;
  if (lane < k) {
    const double f = v[1 + lane], g = v[1 + k + lane], t = t_s[lane];
    double s0 = 0.0, s1 = 0.0;   // two chains
    int i2 = 0;
    for (; i2 + 1 < k; i2 += 2) {
      s0 += gt_s[lane][i2];
      s1 += gt_s[lane][i2 + 1];
    }
    if (i2 < k) s0 += gt_s[lane][i2];
    const double t2 = (g + sigma * f) - (s0 + s1);
    const double cc = beta0 * t - t2 * ti_s[lane];   // (beta_lmp - sigma) t - T^-1 t2
    gt = g * t;
    fc = f * cc;
    lc[lane] = (float)cc;   // Phi columns take c, C Phi columns -t
    lc[k + lane] = -(float)t;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    gt += __shfl_xor_sync(0xffffffffu, gt, o);
    fc += __shfl_xor_sync(0xffffffffu, fc, o);
  }
  if (lane != 0) return;
  double rho = k > 0 ? rr - gt + fc : rr;
  if (lrn) rho = (double)la * rho + v[2 * k + 1];   // r^T (a P^-1 + S S) r = a r^T P^-1 r + u^T u
  pr.betaf[pos] = first ? 0.f : (float)(rho / rho0);
  sd[kRho] = rho;
  sd[kFirst] = 0.0;
  next[at] = (int32_t)j;
  src[at] = (int32_t)pos;
}

// Step 5: p = bf16(r - (C Phi) t + Phi c + beta p) for the running systems, from
// the old position's direction to the new one's (two buffers, or one and the
// memory of y: a workspace without room for the second one).  A warp owns 64
// rows (two consecutive ones per lane) and holds [Phi | C Phi] of its rows in
// registers while it runs over the CTA's systems, four at a time so that their
// loads overlap: 4 k FMAs a lane and system with the coefficients as
// broadcasts, no staging.  (Staging a transposed copy of 512 rows per CTA in
// shared memory, read per system: 14.4 us a launch at 4096 rows, 52 us at 65,536.)
// K: columns of Phi held.
// learned != 0: a learned system takes z = a (r - (C Phi) t + Phi c) + S u.
constexpr int kDirRows = 2;   // consecutive rows per lane
template <int K>
__global__ void __launch_bounds__(kVecThreads) k_tpcg_direction(const ProblemDev* dpr, const int32_t* list,
                                                                const int32_t* src, const __nv_bfloat16* Pold,
                                                                __nv_bfloat16* Pnew, int group, int learned, int it) {
  constexpr int kBatch = 4;
  grid_dependency_wait();
  const ProblemDev& pr = *dpr;
  const int k = pr.kR;
  const int64_t dp = pr.d_pad;
  const int64_t count = pr.nactive[(it + 1) % 3];   // the list the scalars kernel just built
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t g0 = (int64_t)blockIdx.y * group;
  if (g0 >= count) return;
  __shared__ float4 tc4[kMaxGroup][2 * K / 4];   // per system: c (Phi coefficients), then -t (C Phi)
  __shared__ int32_t sys[kMaxGroup], from[kMaxGroup];
  __shared__ float bes[kMaxGroup];
  __shared__ float las[kMaxGroup], ltap[kMaxGroup][kLatBins];   // learned systems: a (0: not learned) and taps
  if (threadIdx.x < kMaxGroup) {
    const int64_t pos = g0 + threadIdx.x;
    const bool on = (int)threadIdx.x < group && pos < count;
    const int j = on ? list[pos] : -1, f = on ? src[pos] : 0;
    sys[threadIdx.x] = j;
    from[threadIdx.x] = f;
    bes[threadIdx.x] = on ? pr.betaf[f] : 0.f;
    float la = 0.f;
    if (learned && on && pr.learn_on[j] == 1) {
      const int64_t q = j < pr.mean_sys ? pr.Q : (j - pr.mean_sys) / pr.N;
      la = pr.learn_coef[q * kLearnOut];
      for (int b = 0; b < kLatBins; ++b) ltap[threadIdx.x][b] = pr.learn_coef[q * kLearnOut + 1 + b];
    }
    las[threadIdx.x] = la;
  }
  __syncthreads();
  float* tcf = reinterpret_cast<float*>(tc4);
  for (int e = threadIdx.x; e < group * 2 * K; e += kVecThreads) {
    const int s = e / (2 * K), m = e % (2 * K);
    float v = 0.f;
    if (sys[s] >= 0) {
      const float* lc = pr.lcoef + (int64_t)from[s] * 2 * kMaxK;
      if (m < K) v = m < k ? lc[m] : 0.f;
      else v = m - K < k ? lc[k + m - K] : 0.f;
    }
    tcf[e] = v;
  }
  const int64_t chunk = (int64_t)blockIdx.x * kVecWarps + warp;
  const bool mine = chunk < dp / (32 * kDirRows);
  const int64_t a = chunk * 32 * kDirRows + lane * kDirRows;
  float c[2 * K][kDirRows];   // loaded while the coefficients are on their way to shared memory
#pragma unroll
  for (int m = 0; m < 2 * K; ++m) {
    const int mm = m < K ? m : k + (m - K);
    const bool in = mine && (m < K ? m < k : m - K < k);
#pragma unroll
    for (int i = 0; i < kDirRows; ++i) c[m][i] = 0.f;
    if (in) {
      const float* col = reinterpret_cast<const float*>(pr.phiT) + (int64_t)mm * dp + a;
      const float2 t = ld_settled(reinterpret_cast<const float2*>(col));
      c[m][0] = t.x;
      c[m][1] = t.y;
    }
  }
  __syncthreads();
  if (!mine) return;
#pragma unroll 1
  for (int s0 = 0; s0 < group; s0 += kBatch) {
    float z[kBatch][kDirRows];
    uint32_t pw[kBatch];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int j = sys[s0 + b];
      if (j < 0) continue;
      const int64_t e = (int64_t)j * dp + a;
      const float2 r = *reinterpret_cast<const float2*>(pr.Rv + e);
      z[b][0] = r.x;
      z[b][1] = r.y;
      pw[b] = *reinterpret_cast<const uint32_t*>(Pold + from[s0 + b] * dp + a);
    }
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int s = s0 + b, j = sys[s];
      if (j < 0) continue;
#pragma unroll
      for (int q = 0; q < 2 * K / 4; ++q) {
        const float4 c4 = tc4[s][q];   // four coefficients (a broadcast load)
        const float cq[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int i = 0; i < kDirRows; ++i) z[b][i] = fmaf(c[4 * q + u][i], cq[u], z[b][i]);
      }
      const float be = bes[s], la = las[s];
#pragma unroll
      for (int i = 0; i < kDirRows; ++i) {
        if (la > 0.f) {   // z = a P^-1 r + S u
          const int32_t* nb = pr.lat_nbr + (a + i) * kLatPts;
          const float* u = pr.learn_u + (int64_t)j * dp;
          float su = 0.f;
#pragma unroll
          for (int n = 0; n < kLatPts; ++n) su = fmaf(ltap[s][lat_bin(n)], ld_settled(u + nb[n]), su);
          z[b][i] = fmaf(la, z[b][i], su);
        }
        const uint32_t w = pw[b];
        const float p = __uint_as_float((i & 1) ? (w & 0xffff0000u) : (w << 16));
        // beta = 0 (a first direction): the old position holds nothing of this system
        z[b][i] = a + i < pr.d ? (be != 0.f ? fmaf(be, p, z[b][i]) : z[b][i]) : 0.f;
      }
      *reinterpret_cast<__nv_bfloat162*>(Pnew + (g0 + s) * dp + a) = __floats2bfloat162_rn(z[b][0], z[b][1]);
    }
  }
}

// Systems per CTA of the direction kernel (a multiple of its batch of four):
// enough that a CTA's load of [Phi | C Phi] (80 bytes a row) is small beside
// its systems' vectors (8 bytes a row each), few enough that small problems
// still give every SM about 12 warps.
int dir_group(int64_t nchunk, int64_t count, int sms) {
  const int64_t g = (nchunk * count + 12 * sms - 1) / (12 * (int64_t)sms);
  return (int)std::min<int64_t>(std::max<int64_t>((g + 3) / 4 * 4, 4), kMaxGroup);
}

}  // namespace

// Runs the PCG of one BF16 problem (host copy p, device copy dp) to
// convergence or the iteration cap.  The kernels take the number of running
// systems from the device; the host needs it only to size the launches and to
// stop, so it reads it one iteration late: iteration `it` is launched with the
// count after iteration it - 2, while iteration it - 1 runs (the count never
// grows), and the call that finds nothing running costs one iteration of
// empty launches.  cap != NULL: records the Krylov samples of its systems at
// iterations 1..cap->K and stops after K iterations, without the learned term.
static int tile_pcg_loop(const ProblemDev& p, const ProblemDev* dp, cudaStream_t st, double* mm_ms, int* mm_count,
                         const TileCapture* cap) {
  const int64_t J = p.nsys;
  if (J < 1) return 0;
  AuxStream* aux = aux_stream();   // NULL: the counts are read on st, behind the iteration in flight
  cudaEvent_t ev[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};   // matvec begin and end, iterations in turn
  struct Destroy {
    cudaEvent_t (*e)[2];
    ~Destroy() {
      for (int i = 0; i < 4; ++i)
        if (e[i / 2][i % 2]) cudaEventDestroy(e[i / 2][i % 2]);
    }
  } destroy{ev};
  for (int i = 0; mm_ms && i < 4; ++i)
    if (cudaEventCreate(&ev[i / 2][i % 2]) != cudaSuccess) {
      cudaGetLastError();
      return INFO_ESRF_ERR_CUDA;
    }
  const bool wide = p.kR > 12;   // 24 columns of Phi in registers
  const int nsub = (int)((p.d_pad + kDotRows - 1) / kDotRows);
  const int64_t dchunks = p.d_pad / 64;
  const dim3 gsys((unsigned)((J + 127) / 128));
  const dim3 gall((unsigned)((J * p.d_pad + 255) / 256));
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return INFO_ESRF_ERR_CUDA;
  TileMmArgs ta{};
  ta.rowptr = p.rowptr;
  ta.colblk = p.colblk;
  ta.sigma = p.sigmaf;
  ta.Y = p.Yv;
  ta.pty = p.pty;
  ta.status = p.status;
  ta.d_pad = p.d_pad;
  ta.J = (int32_t)J;
  ta.nrt = p.nrt;
  ta.pty_by_system = 1;
  int maxit = p.fixed_iters > 0 ? p.fixed_iters : p.max_iter;
  if (cap) maxit = cap->K;
  // the learned term is possible when the problem has a model and its tables
  bool learned = !cap && p.learned_model && p.learn_on && p.lat_info;
  const bool fused_alpha = p.nrt <= kFusedAlpha;
  const size_t usm = (size_t)2 * p.kR * kDotRows * sizeof(float);
  static thread_local int raised = -1;
  if (raised != dev) {
    const int mx = 2 * kMaxK * kDotRows * (int)sizeof(float);
    if (cudaFuncSetAttribute(k_tpcg_update<1, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx) != cudaSuccess ||
        cudaFuncSetAttribute(k_tpcg_update<1, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx) != cudaSuccess ||
        cudaFuncSetAttribute(k_tpcg_update<2, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx) != cudaSuccess)
      return INFO_ESRF_ERR_CUDA;
    raised = dev;
  }
  // The lists of running systems and of their positions before, in turn.
  int32_t* lists[2] = {p.alist, p.alist + J};
  int32_t* srcs = p.alist + 2 * J;
  // mode 0: the dot products of r alone; 1, 2: the update (2 forms alpha in it)
  auto update = [&](int mode, const int32_t* list, int64_t count, int it) {
    // two systems per thread (half the reads of [Phi | C Phi]) once that still
    // gives every SM two CTAs; 64 dot values (k > 15) leave registers for one
    const __nv_bfloat16* P = p.Pcur(it);
    const int spt = p.kR <= 15 && nsub * count >= 32 * (int64_t)sms ? 2 : 1;
    const int64_t groups = (count + kUpdSlots * spt - 1) / (kUpdSlots * spt), layers = (groups + 65534) / 65535;
    const dim3 grid((unsigned)nsub, (unsigned)((groups + layers - 1) / layers), (unsigned)layers);
    if (p.kR > 15) launch_overlapped(k_tpcg_update<2, 1>, grid, kUpdThreads, usm, st, dp, mode, list, P, it);
    else if (spt == 2) launch_overlapped(k_tpcg_update<1, 2>, grid, kUpdThreads, usm, st, dp, mode, list, P, it);
    else launch_overlapped(k_tpcg_update<1, 1>, grid, kUpdThreads, usm, st, dp, mode, list, P, it);
  };
  auto direction = [&](const int32_t* list, int64_t count, int it) {
    const int group = dir_group(dchunks, count, sms);
    const dim3 grid((unsigned)((dchunks + kVecWarps - 1) / kVecWarps), (unsigned)((count + group - 1) / group));
    const int32_t* from = srcs;
    const __nv_bfloat16* Pold = p.Pcur(it);
    __nv_bfloat16* Pnew = p.Pnext(it);
    const int lrn = learned ? 1 : 0;
    auto kernel = wide ? k_tpcg_direction<24> : k_tpcg_direction<12>;
    launch_overlapped(kernel, grid, kVecThreads, 0, st, dp, list, from, Pold, Pnew, group, lrn, it);
    // one direction buffer: y, where they were formed, is free until the next matvec (3.34 ms
    // for 3.13 at 961 systems x 960 observations, the same bits)
    if (!p.Pdir1)
      cudaMemcpyAsync(p.Pdir, p.Yv, (size_t)count * p.d_pad * sizeof(__nv_bfloat16), cudaMemcpyDeviceToDevice, st);
  };
  // iteration 0, the first direction of every running system: r = b, z = M r, p = z
  auto start = [&]() {
    update(0, nullptr, J, 0);
    if (learned) launch_tile_learn_u(p, dp, nullptr, J, nsub, 0, st);
    k_tpcg_scalars<<<(unsigned)J, kScalThreads, 0, st>>>(dp, nsub, maxit <= 0 ? 1 : 0, nullptr, lists[1], srcs, 0);
    if (aux) cudaEventRecord(aux->counted[0], st);
    direction(lists[1], J, 0);
    note_launches(3);
  };
  // counts[it + 1] (and the status word) after iteration it, read on a stream of
  // its own so that the main stream keeps running and the host waits for nothing
  // else.  (Iteration it + 1 leaves the slot alone: on st the value is the same.)
  int32_t host[4] = {0, 0, 0, 0};
  auto read_counts = [&](int it) -> int {
    const cudaStream_t rs = aux ? aux->count : st;
    if ((aux && cudaStreamWaitEvent(rs, aux->counted[it & 1], 0) != cudaSuccess) ||
        cudaMemcpyAsync(host, p.nactive, sizeof(host), cudaMemcpyDeviceToHost, rs) != cudaSuccess ||
        cudaStreamSynchronize(rs) != cudaSuccess)
      return INFO_ESRF_ERR_CUDA;
    return 0;
  };
  auto iterate = [&]() -> int {
    int64_t bound = J;   // systems that iteration it may run
    int timed = -1;      // the iteration whose matvec events await reading
    auto read_time = [&]() -> int {
      if (timed < 0) return 0;
      float ms = 0.f;
      if (cudaEventSynchronize(ev[timed & 1][1]) != cudaSuccess) return INFO_ESRF_ERR_CUDA;
      if (cudaEventElapsedTime(&ms, ev[timed & 1][0], ev[timed & 1][1]) == cudaSuccess) {
        *mm_ms += ms;
        ++*mm_count;
      }
      timed = -1;
      return 0;
    };
    for (int it = 1; it <= maxit; ++it) {
      if (it >= 2) {
        if (read_counts(it - 2) || (mm_ms && read_time())) return INFO_ESRF_ERR_CUDA;
        if (host[3] & (kStatTimeout | kStatTileOverflow)) return 0;
        bound = host[(it - 1) % 3];   // running in iteration it - 1
        if (bound == 0) return 0;     // it ran nothing, and its matvec is not counted
        if (mm_ms) timed = it - 1;
      }
      const int32_t* list = lists[it & 1];
      int32_t* next = lists[(it + 1) & 1];
      ta.P = p.Pcur(it);
      ta.count = p.nactive + it % 3;
      ta.list = list;
      ta.J_run = (int32_t)bound;
      if (mm_ms) cudaEventRecord(ev[it & 1][0], st);
      if (launch_tile_mm(ta, p.Chi, p.Clo, p.tile_cap, st) != 0) return INFO_ESRF_ERR_CUDA;
      if (mm_ms) cudaEventRecord(ev[it & 1][1], st);
      if (cap) launch_tile_capture_record(p, dp, *cap, it, list, st);
      if (!fused_alpha) {
        k_tpcg_alpha<<<(unsigned)((32 * bound + 255) / 256), 256, 0, st>>>(dp, it, list);
        note_launches(1);
      }
      update(fused_alpha ? 2 : 1, list, bound, it);
      if (learned) launch_tile_learn_u(p, dp, list, bound, nsub, it, st);
      launch_overlapped(k_tpcg_scalars, dim3((unsigned)bound), kScalThreads, 0, st, dp, nsub, it == maxit ? 1 : 0, list,
                        next, srcs, it);
      if (aux) cudaEventRecord(aux->counted[it & 1], st);
      direction(next, bound, it);
      note_launches(3);
    }
    if (mm_ms && maxit >= 1) {   // the cap was reached: the last two matvecs, if they ran anything
      if (read_time()) return INFO_ESRF_ERR_CUDA;
      if (read_counts(maxit - 1)) return INFO_ESRF_ERR_CUDA;
      if (host[maxit % 3] > 0) {
        timed = maxit;
        if (read_time()) return INFO_ESRF_ERR_CUDA;
      }
    }
    return 0;
  };
  k_tpcg_init<<<gall, 256, 0, st>>>(dp, 0, learned ? 1 : 0);
  k_tpcg_phit<<<(unsigned)((p.d_pad + 255) / 256), 256, 0, st>>>(dp);
  note_launches(2);
  if (learned) {   // systems that use the term (none: the plain loop)
    int32_t nl = 0;
    if (cudaMemcpyAsync(&nl, p.lat_info + 8, sizeof(int32_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return INFO_ESRF_ERR_CUDA;
    learned = nl > 0;
  }
  start();
  int rc = iterate();
  if (rc) return rc;
  if (learned) {
    // plain PCG for the learned systems that broke down or hit the cap
    int32_t retries = 0;
    if (cudaMemcpyAsync(&retries, p.lat_info + 7, sizeof(int32_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return INFO_ESRF_ERR_CUDA;
    if (retries > 0) {
      k_tpcg_retry_vectors<<<gall, 256, 0, st>>>(dp);
      k_tpcg_init<<<gsys, 128, 0, st>>>(dp, 1, 0);
      note_launches(2);
      start();
      rc = iterate();
      if (rc) return rc;
    }
  }
  return cudaGetLastError() == cudaSuccess ? 0 : INFO_ESRF_ERR_CUDA;
}

int run_tile_pcg(const ProblemDev& p, const ProblemDev* dp, cudaStream_t st, double* mm_ms, int* mm_count) {
  return tile_pcg_loop(p, dp, st, mm_ms, mm_count, nullptr);
}

int run_tile_pcg_capture(const ProblemDev& p, const ProblemDev* dp, const TileCapture& cap, float* Z, float* feat,
                         cudaStream_t st) {
  const int rc = tile_pcg_loop(p, dp, st, nullptr, nullptr, &cap);
  if (rc) return rc;
  launch_tile_capture_finish(p, dp, cap, Z, feat, st);
  return cudaGetLastError() == cudaSuccess ? 0 : INFO_ESRF_ERR_CUDA;
}

}  // namespace infoesrf
