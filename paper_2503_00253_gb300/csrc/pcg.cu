// a5-a8: persistent batched shifted PCG over every (quadrature node, member)
// system of every problem, plus the mean system (App. E, Eq.
// normalized_linear_solve; Golub & Van Loan Alg. 11.5.1):
//
//     C_q u = b,   C_q = (s_q + 1) I + C,   C = R^-1/2 (L_oo o W W^T) R^-1/2,
//     b = R^-1/2 w_f^(i)  (perturbation)   or   R^-1/2 (y - H mu)  (mean, s = 0).
//
// All systems share the band of C, formed once per analysis, so the matvec
// is a banded sparse-times-dense product over a group of JT systems that
// share one shift.  Each CTA owns one group at a time: its PCG vectors sit
// in shared memory as far as they fit (in a private global slice otherwise),
// so a group iterates to convergence without any grid-wide synchronization.
// Groups come from an atomic queue, so CTAs that finish early take more.
//
// Preconditioner: the limited-memory preconditioner of App. E,
//   P_q^-1 = (I - Phi T^-1 Phi^T C_q)(I - C_q Phi T^-1 Phi^T) + beta Phi T^-1 Phi^T,
// applied with f = Phi^T r, g = A^T r (A = C Phi) and the k x k matrix
// G_q = (C_q Phi)^T (C_q Phi):  t = T^-1 f,  t2 = g + sigma f - G_q t,
// c = (beta - sigma) t - T^-1 t2,  z = r - A t + Phi c,  r^T z = r^T r - g.t + f.c.
// So f, g and r^T r come out of one pass over the residual.
//
// Scalars (rho, alpha, beta, norms, the k x k preconditioner algebra) are FP64,
// one warp per system; dot products of FP32 vectors are accumulated as
// float-float pairs.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace infoesrf {

// Layout of a group's vectors: [row][JT], a row's JT systems side by side.  A
// work item is VL consecutive systems of a row (16 bytes of FP32, one FP64
// value); item i = row G + g with G = JT / VL, so consecutive items are
// consecutive in memory and a thread that strides by a multiple of G always
// serves the same systems g VL .. g VL + VL - 1.
//
// FP64: one value per item, because the FP64 pipe (about two lanes per clock
// and SM) is the bound and only needs every warp to carry some of the work.
// FP32: four, so that an entry of C serves four systems per 16-byte read of p.
constexpr int kPcgThreads = 512;
constexpr int kPcgWarps = kPcgThreads / 32;
template <typename T> struct PcgVec;
template <> struct PcgVec<float> { static constexpr int VL = 4; };
template <> struct PcgVec<double> { static constexpr int VL = 1; };
// Systems per group: two items a row (an entry of C and a column of Phi serve
// both); in FP64 one for problems of few groups (pcg_jt).
template <typename T> constexpr int kJTWide = 2 * PcgVec<T>::VL;
template <typename T> constexpr int kJTNarrow = sizeof(T) == 8 ? 1 : kJTWide<T>;

template <typename T>
struct Item {
  T v[PcgVec<T>::VL];
};
__device__ __forceinline__ Item<float> ld_item(const float* p) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  return Item<float>{{t.x, t.y, t.z, t.w}};
}
__device__ __forceinline__ Item<double> ld_item(const double* p) { return Item<double>{{*p}}; }
__device__ __forceinline__ void st_item(float* p, const Item<float>& a) {
  *reinterpret_cast<float4*>(p) = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
}
__device__ __forceinline__ void st_item(double* p, const Item<double>& a) { *p = a.v[0]; }

struct GroupInfo {
  int prob;
  int lanes;     // active systems in this group
  int i0;        // first member (perturbation groups)
  int q;         // quadrature index, -1 for the mean system
};

__device__ __forceinline__ GroupInfo decode_group(const ProblemDev* tab, int count, int gg) {
  GroupInfo gi;
  int lo = 0, hi = count - 1;   // the last problem whose group_base is at most gg
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tab[mid].group_base <= gg) lo = mid;
    else hi = mid - 1;
  }
  const ProblemDev& pr = tab[lo];
  gi.prob = lo;
  const int lg = gg - pr.group_base;
  if (lg < pr.mean_sys) {         // the mean system comes first (hardest shift)
    gi.q = -1;
    gi.i0 = 0;
    gi.lanes = 1;
  } else {
    const int pg = lg - pr.mean_sys;
    gi.q = pg / pr.groups_per_q;
    gi.i0 = (pg % pr.groups_per_q) * pr.JT;
    const int left = (int)pr.N - gi.i0;
    gi.lanes = left < pr.JT ? left : pr.JT;
  }
  return gi;
}

template <typename T, int KMAX, int JT>
struct PcgShared {
  alignas(16) T coef[2 * KMAX][JT];        // direction: c for the Phi columns, -t for the C Phi columns
  T red[4 * kPcgWarps][JT];                // projections: [set][4 nq columns]
  double Gq[KMAX * KMAX + 1];
  double ith[KMAX + 1];                    // 1 / (theta + sigma)
  double rho[JT], bn2[JT], rr[JT];
  T alpha[JT], beta[JT];
  float wpf[JT][kPcgWarps][2];
  double wpd[JT][kPcgWarps];
  double ts[JT][KMAX + 1];
  int active[JT], iters[JT];
  double sigma, beta_lmp;
};

// Sums acc over the lanes of a warp that serve the same systems (lane mod G)
// and writes the warp's partial of each system.
template <typename T, int KMAX, int JT>
__device__ __forceinline__ void warp_partials(PcgShared<T, KMAX, JT>& sh, const DotAcc<T> (&acc)[PcgVec<T>::VL],
                                              int warp, int lane) {
  constexpr int VL = PcgVec<T>::VL, G = JT / VL;
#pragma unroll
  for (int v = 0; v < VL; ++v) {
    if constexpr (sizeof(T) == 4) {
      float hi = acc[v].hi, lo = acc[v].lo;
#pragma unroll
      for (int o = 16; o >= G; o >>= 1) {
        const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
        const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
        ff_merge(hi, lo, h2, l2);
      }
      if (lane < G) {
        sh.wpf[lane * VL + v][warp][0] = hi;
        sh.wpf[lane * VL + v][warp][1] = lo;
      }
    } else {
      double s = acc[v].value();
#pragma unroll
      for (int o = 16; o >= G; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane < G) sh.wpd[lane * VL + v][warp] = s;
    }
  }
}

// Sum of the warps' partials of system j, by one warp.  Every lane returns lane
// 0's value: the callers branch on it, and all lanes must take the same way
// (the low parts of a float-float butterfly may differ between lanes).
template <typename T, int KMAX, int JT>
__device__ __forceinline__ double combine_partials(const PcgShared<T, KMAX, JT>& sh, int j, int lane) {
  static_assert(kPcgWarps <= 32, "one lane per warp partial");
  double s;
  if constexpr (sizeof(T) == 4) {
    float hi = lane < kPcgWarps ? sh.wpf[j][lane][0] : 0.f, lo = lane < kPcgWarps ? sh.wpf[j][lane][1] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
      const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
      ff_merge(hi, lo, h2, l2);
    }
    s = (double)hi + (double)lo;
  } else {
    s = lane < kPcgWarps ? sh.wpd[j][lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  return __shfl_sync(0xffffffffu, s, 0);
}

// Where a group's vectors live, by the problem's size: level 0 all four in
// shared memory, 1 the direction p (which the matvec gathers) there and the
// others in the CTA's global slice, 2 all in the slice.
struct PcgLayout {
  int level;
  size_t pvec, vec;   // elements of p (rows padded by a quarter in FP32) and of the others
};

// Row of p in its buffer: FP32 rows of 32 bytes get one empty row after every
// four, so that rows four apart (the e-th columns of neighbouring row quads)
// start in different banks.
template <typename T>
__host__ __device__ __forceinline__ int64_t p_row(int64_t a) {
  return sizeof(T) == 4 ? a + (a >> 2) : a;
}

constexpr size_t kPcgSmem = 200 * 1024;   // dynamic shared memory of a CTA (one CTA per SM)
constexpr int kPcgChunk = 1024;           // rows of r staged at a time for the projections (levels 1 and 2)

template <typename T>
__host__ __device__ __forceinline__ PcgLayout pcg_layout(int64_t d, int JT) {
  PcgLayout l;
  l.vec = (size_t)d * JT;
  l.pvec = (size_t)p_row<T>(d + 3) * JT;
  const size_t chunk = (size_t)kPcgChunk * JT * sizeof(T);
  if ((l.pvec + 3 * l.vec) * sizeof(T) <= kPcgSmem) l.level = 0;
  else if (l.pvec * sizeof(T) + chunk <= kPcgSmem) l.level = 1;
  else l.level = 2;
  return l;
}

// One group to convergence, by all threads of the CTA.
template <typename T, int KMAX, int JT>
__device__ __forceinline__ void solve_group(const ProblemDev& pr, const GroupInfo& gi, T* sm, T* slice,
                                            PcgShared<T, KMAX, JT>& sh) {
  constexpr int VL = PcgVec<T>::VL, G = JT / VL;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = tid % G;   // which systems of a row this thread serves, in every item loop
  const int d = (int)pr.d;
  const int64_t N = pr.N;
  const int k = pr.kR < KMAX ? pr.kR : KMAX;
  const PcgLayout lay = pcg_layout<T>(d, JT);
  T* vp = lay.level <= 1 ? sm : slice + 3 * lay.vec;
  T* vr = lay.level == 0 ? sm + lay.pvec : slice;
  T* vy = vr + lay.vec;
  T* vx = vy + lay.vec;
  T* rbuf = lay.level == 0 ? vr : (lay.level == 1 ? sm + lay.pvec : sm);   // rows of r under projection
  const int crows = lay.level == 0 ? d : kPcgChunk;
  const T* __restrict__ val = reinterpret_cast<const T*>(pr.oo_val);
  const int32_t* __restrict__ col = pr.oo_col;
  const T* __restrict__ PhiT = reinterpret_cast<const T*>(pr.phiT);   // [2 k][d]
  const T* __restrict__ W = reinterpret_cast<const T*>(pr.W);

  // ---- group setup: shift, LMP constants, G_q ----
  if (tid == 0) {
    const double s = gi.q < 0 ? 0.0 : pr.s[gi.q];
    sh.sigma = s + 1.0;
    sh.beta_lmp = sh.sigma + pr.scal[1];
  }
  __syncthreads();
  const double sigma = sh.sigma;
  const T sigma_t = to_t<T>(sigma);
  for (int e = tid; e < k * k; e += kPcgThreads) {
    const int i = e / k, j = e % k;
    const int kk = pr.kR;   // gram matrices are stored with the problem's k
    const int ge = i * kk + j, gt = j * kk + i;
    // G_q = A^T A + sigma (A^T Phi + Phi^T A) + sigma^2 Phi^T Phi
    sh.Gq[e] = pr.gram[2 * kk * kk + ge] + sigma * (pr.gram[kk * kk + ge] + pr.gram[kk * kk + gt]) +
               sigma * sigma * pr.gram[ge];
  }
  for (int m = tid; m < k; m += kPcgThreads) sh.ith[m] = 1.0 / (pr.theta[m] + sigma);
  if (tid < JT) {
    sh.active[tid] = tid < gi.lanes;
    sh.iters[tid] = 0;
    sh.beta[tid] = T(0);
    sh.rr[tid] = 0.0;
    sh.alpha[tid] = T(0);
  }

  // ---- x = 0, r = b, p = 0 ----
  for (int e = tid; e < d * JT; e += kPcgThreads) {
    const int a = e / JT, j = e % JT;
    T b = T(0);
    if (j < gi.lanes) {
      if (gi.q < 0) b = to_t<T>(pr.bmean[a]);
      else b = W[a * N + gi.i0 + j] * to_t<T>(pr.rinv[a]);
    }
    vr[e] = b;
    vx[e] = T(0);
    vp[p_row<T>(a) * JT + j] = T(0);
  }
  __syncthreads();

  bool first = true;
  const int maxit = pr.fixed_iters > 0 ? pr.fixed_iters : pr.max_iter;
  const int nq = (2 * k + 3) / 4;              // column quads of [Phi | C Phi]
  const int sets = nq > 0 ? kPcgWarps / nq : 1;   // warps per quad
  const int quad = nq > 0 ? warp % nq : 0, set = nq > 0 ? warp / nq : 0;

  // The update x += alpha p, r -= alpha y (not on the first call), then
  // r^T r, f = Phi^T r and g = A^T r, in one pass: rows of r go through
  // shared memory, where warp (quad, set) projects them on its four columns
  // with 4 JT register accumulators, lanes over rows (coalesced columns).
  // Then the scalars, one warp per system.
  auto residual_pass = [&]() {
    DotAcc<T> rr[VL];
    T acc[4][JT];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < JT; ++j) acc[i][j] = T(0);
    T al[VL];
#pragma unroll
    for (int v = 0; v < VL; ++v) al[v] = sh.alpha[g * VL + v];
    for (int c0 = 0; c0 < d; c0 += crows) {
      const int nr = d - c0 < crows ? d - c0 : crows;
      // kU items at once: their loads are all in flight before the first use
      // (levels 1 and 2 stream the vectors from L2)
      constexpr int kU = 2;
      for (int it0 = tid; it0 < nr * G; it0 += kU * kPcgThreads) {
        Item<T> r[kU], y[kU], x[kU], p[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const int it = it0 + u * kPcgThreads;
          if (it >= nr * G) continue;
          const int64_t o = ((int64_t)c0 * G + it) * VL;
          r[u] = ld_item(vr + o);
          if (first) continue;
          y[u] = ld_item(vy + o);
          x[u] = ld_item(vx + o);
          p[u] = ld_item(vp + p_row<T>(c0 + it / G) * JT + g * VL);
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const int it = it0 + u * kPcgThreads;
          if (it >= nr * G) continue;
          const int64_t o = ((int64_t)c0 * G + it) * VL;
          if (!first) {
#pragma unroll
            for (int v = 0; v < VL; ++v) {
              x[u].v[v] += al[v] * p[u].v[v];
              r[u].v[v] -= al[v] * y[u].v[v];
            }
            st_item(vx + o, x[u]);
            st_item(vr + o, r[u]);
          }
          if (lay.level != 0) st_item(rbuf + (int64_t)it * VL, r[u]);
#pragma unroll
          for (int v = 0; v < VL; ++v) rr[v].add_prod(r[u].v[v], r[u].v[v]);
        }
      }
      if (nq == 0) continue;
      __syncthreads();
      if (set < sets) {
        const int m0 = 4 * quad;
#pragma unroll 2
        for (int a = lane + 32 * set; a < nr; a += 32 * sets) {
          T rv[JT];
#pragma unroll
          for (int u = 0; u < G; ++u) {
            const Item<T> t = ld_item(rbuf + (int64_t)a * JT + u * VL);
#pragma unroll
            for (int v = 0; v < VL; ++v) rv[u * VL + v] = t.v[v];
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const T ph = m0 + i < 2 * k ? PhiT[(int64_t)(m0 + i) * d + c0 + a] : T(0);
#pragma unroll
            for (int j = 0; j < JT; ++j) acc[i][j] += ph * rv[j];
          }
        }
      }
      if (c0 + crows < d) __syncthreads();   // the next chunk overwrites the buffer
    }
    warp_partials<T, KMAX, JT>(sh, rr, warp, lane);
    if (nq > 0 && set < sets) {
      // reduce-scatter the 4 JT sums over the warp: first halve the values
      // held per lane, then sum the lanes that hold the same value
      constexpr int V = 4 * JT;   // 32 (FP32), 8 or 4 (FP64)
      T* v = &acc[0][0];
      int idx = 0;
#pragma unroll
      for (int off = 16, w = V / 2; w >= 1; off >>= 1, w >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < w; ++i) {
          const T send = up ? v[i] : v[i + w];
          const T keep = up ? v[i + w] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
        if (up) idx += w;
      }
#pragma unroll
      for (int off = 16 / V; off >= 1; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
      if ((lane & (32 / V - 1)) == 0) sh.red[set * 4 * nq + 4 * quad + idx / JT][idx % JT] = v[0];
    }
    __syncthreads();
    if (warp < JT) {
      const int j = warp;
      const double rr_j = combine_partials<T, KMAX, JT>(sh, j, lane);
      const bool was_active = sh.active[j] != 0;
      const double bn2 = first ? rr_j : sh.bn2[j];
      __syncwarp();   // lane 0 writes both below
      bool act = was_active;
      if (act && pr.fixed_iters <= 0 && !(rr_j > pr.tol * pr.tol * bn2)) act = false;
      if (act && (!(rr_j > 0.0) || !isfinite(rr_j))) act = false;
      double rho = rr_j;
      if (k > 0 && act) {
        T fs = T(0), gs = T(0);
        if (lane < k)
          for (int s = 0; s < sets; ++s) {
            fs += sh.red[s * 4 * nq + lane][j];
            gs += sh.red[s * 4 * nq + k + lane][j];
          }
        const double f = (double)fs, gg2 = (double)gs;
        const double ith = lane < k ? sh.ith[lane] : 0.0;
        const double t = f * ith;
        if (lane < k) sh.ts[j][lane] = t;
        __syncwarp();
        double a0 = 0.0, a1 = 0.0;   // G_q t, two chains
        if (lane < k) {
          int i2 = 0;
          for (; i2 + 1 < k; i2 += 2) {
            a0 += sh.Gq[lane * k + i2] * sh.ts[j][i2];
            a1 += sh.Gq[lane * k + i2 + 1] * sh.ts[j][i2 + 1];
          }
          if (i2 < k) a0 += sh.Gq[lane * k + i2] * sh.ts[j][i2];
        }
        const double t2 = gg2 + sigma * f - (a0 + a1);
        const double c = (sh.beta_lmp - sigma) * t - t2 * ith;
        double df = lane < k ? f * c - gg2 * t : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) df += __shfl_xor_sync(0xffffffffu, df, o);
        rho = rr_j + df;
        if (lane < k) {
          sh.coef[lane][j] = to_t<T>(c);
          sh.coef[k + lane][j] = to_t<T>(-t);
        }
      }
      if (lane == 0) {
        if (first) sh.bn2[j] = rr_j;
        if (!act) {
          sh.beta[j] = T(0);
        } else {
          sh.beta[j] = first ? T(0) : to_t<T>(rho / sh.rho[j]);
          sh.rho[j] = rho;
        }
        if (was_active || first) sh.rr[j] = rr_j;
        sh.active[j] = act;
      }
    }
    __syncthreads();
    int any = 0;
#pragma unroll
    for (int j = 0; j < JT; ++j) any |= sh.active[j];
    return any != 0;
  };

  // z = P^-1 r, p = z + beta p (a stopped system keeps its p)
  auto update_direction = [&]() {
    T be[VL];
    bool on[VL];
#pragma unroll
    for (int v = 0; v < VL; ++v) {
      be[v] = sh.beta[g * VL + v];
      on[v] = sh.active[g * VL + v] != 0;
    }
    constexpr int kU = sizeof(T) == 4 ? 4 : 2;   // items side by side: one read of the coefficients serves all
    for (int it = tid; it < d * G; it += kU * kPcgThreads) {
      Item<T> z[kU];
      int a[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int iu = it + u * kPcgThreads;
        a[u] = iu < d * G ? iu / G : 0;
        z[u] = ld_item(vr + (int64_t)a[u] * JT + g * VL);
      }
#pragma unroll 4
      for (int m = 0; m < 2 * k; ++m) {
        const Item<T> c = ld_item(&sh.coef[m][g * VL]);
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const T ph = PhiT[(int64_t)m * d + a[u]];
#pragma unroll
          for (int v = 0; v < VL; ++v) z[u].v[v] += ph * c.v[v];
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        if (it + u * kPcgThreads >= d * G) continue;
        T* pp = vp + p_row<T>(a[u]) * JT + g * VL;
        Item<T> p = ld_item(pp);
#pragma unroll
        for (int v = 0; v < VL; ++v) p.v[v] = on[v] ? z[u].v[v] + be[v] * p.v[v] : p.v[v];
        st_item(pp, p);
      }
    }
    __syncthreads();
  };

  bool run = residual_pass();
  first = false;
  if (run) update_direction();

  // FP32: C by quads of rows where the set-up made them (k_pcg_quads)
  const bool quads = sizeof(T) == 4 && pr.qval && pr.status[2] == 0;
  // items of the matvec, and threads per item: the largest power of two that
  // still covers all items at once (small problems split a row's entries)
  const int items = (quads ? (d + 3) / 4 : d) * G;
  int tpi = 1;
  while (tpi < 16 && 2 * tpi * items <= kPcgThreads) tpi *= 2;
  const int per = 32 / tpi, sub = lane / per, ii = lane % per;

  int it = 0;
  while (run && it < maxit) {
    ++it;
    // ---- y = C_q p, p^T y ----
    DotAcc<T> pap[VL];
    const int iend = (items + per - 1) / per * per;   // whole warps take part in the shuffles
    if constexpr (sizeof(T) == 4) {
      if (quads) {
        const int nb = (d + 3) / 4;
        const float4* __restrict__ qv = reinterpret_cast<const float4*>(pr.qval);
        const int32_t* __restrict__ qc = pr.qcol;
        for (int i = warp * per + ii; i < iend; i += kPcgWarps * per) {
          const bool in = i < items;
          const int blk = in ? i / G : 0;
          float acc[4][VL] = {};
          const int n = in ? pr.qn[blk] : 0;
#pragma unroll 8
          for (int e = sub; e < n; e += tpi) {
            const float4 c = qv[(int64_t)e * nb + blk];
            const Item<T> pb = ld_item(vp + qc[(int64_t)e * nb + blk] + g * VL);
            const float cc[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
            for (int w = 0; w < 4; ++w)
#pragma unroll
              for (int v = 0; v < VL; ++v) acc[w][v] = fmaf(cc[w], pb.v[v], acc[w][v]);
          }
          for (int o = 16; o >= per; o >>= 1)
#pragma unroll
            for (int w = 0; w < 4; ++w)
#pragma unroll
              for (int v = 0; v < VL; ++v) acc[w][v] += __shfl_xor_sync(0xffffffffu, acc[w][v], o);
          if (in && sub == 0) {
#pragma unroll
            for (int w = 0; w < 4; ++w) {
              const int a = 4 * blk + w;
              if (a >= d) break;
              const Item<T> p = ld_item(vp + p_row<T>(a) * JT + g * VL);
              Item<T> y;
#pragma unroll
              for (int v = 0; v < VL; ++v) {
                y.v[v] = fmaf(sigma_t, p.v[v], acc[w][v]);
                pap[v].add_prod(p.v[v], y.v[v]);
              }
              st_item(vy + (int64_t)a * JT + g * VL, y);
            }
          }
        }
      }
    }
    if (!quads) {
      for (int i = warp * per + ii; i < iend; i += kPcgWarps * per) {
        const bool in = i < items;
        const int a = in ? i / G : 0;
        Item<T> acc{};
        const int nnz = in ? pr.oo_nnz[a] : 0;
#pragma unroll 4
        for (int e = sub; e < nnz; e += tpi) {
          const T c = val[(int64_t)e * d + a];
          const int b = col[(int64_t)e * d + a];
          const Item<T> pb = ld_item(vp + p_row<T>(b) * JT + g * VL);
#pragma unroll
          for (int v = 0; v < VL; ++v) acc.v[v] += c * pb.v[v];
        }
        for (int o = 16; o >= per; o >>= 1)
#pragma unroll
          for (int v = 0; v < VL; ++v) acc.v[v] += __shfl_xor_sync(0xffffffffu, acc.v[v], o);
        if (in && sub == 0) {
          const Item<T> p = ld_item(vp + p_row<T>(a) * JT + g * VL);
#pragma unroll
          for (int v = 0; v < VL; ++v) {
            acc.v[v] += sigma_t * p.v[v];
            pap[v].add_prod(p.v[v], acc.v[v]);
          }
          st_item(vy + (int64_t)a * JT + g * VL, acc);
        }
      }
    }
    warp_partials<T, KMAX, JT>(sh, pap, warp, lane);
    __syncthreads();
    if (warp < JT) {
      const int j = warp;
      const double pAp = combine_partials<T, KMAX, JT>(sh, j, lane);
      if (lane == 0) {
        T alpha = T(0);
        if (sh.active[j]) {
          if (pAp > 0.0 && isfinite(pAp)) {
            alpha = to_t<T>(sh.rho[j] / pAp);
            sh.iters[j] = it;
          } else {
            sh.active[j] = 0;
            atomicOr(&pr.status[0], kStatBreakdown);
          }
        }
        sh.alpha[j] = alpha;
      }
    }
    __syncthreads();
    run = residual_pass();
    if (!run) break;
    update_direction();
  }

  // ---- results ----
  // lane j holds system sid0 + j (the mean group has one lane, sid 0)
  const int64_t sid0 = gi.q < 0 ? 0 : pr.mean_sys + (int64_t)gi.q * N + gi.i0;
  T* U = reinterpret_cast<T*>(pr.U);
  for (int j = 0; j < gi.lanes; ++j)
    for (int a = tid; a < d; a += kPcgThreads) U[(sid0 + j) * d + a] = vx[(int64_t)a * JT + j];
  if (tid < gi.lanes) {
    const int64_t sidx = sid0 + tid;
    pr.iters[sidx] = sh.iters[tid];
    const double bn = sh.bn2[tid];
    pr.relres[sidx] = bn > 0 ? sqrt(sh.rr[tid] / bn) : 0.0;
    if (sh.active[tid] && pr.fixed_iters <= 0) atomicOr(&pr.status[0], kStatNotConverged);
  }
  __syncthreads();
}

template <typename T, int KMAX>
__global__ void __launch_bounds__(kPcgThreads, 1)
k_pcg(const ProblemDev* tab, int count, int total_groups, int32_t* counter, T* gscratch,
      int64_t scratch_stride, uint64_t band_mask, const int32_t* band_fb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ union Shared {
    PcgShared<T, KMAX, kJTWide<T>> wide;
    PcgShared<T, KMAX, kJTNarrow<T>> narrow;
    __device__ Shared() {}
  } sh;
  __shared__ int s_group;
  const int tid = threadIdx.x;
  T* sm = reinterpret_cast<T*>(smem_raw);
  T* slice = gscratch + (int64_t)blockIdx.x * scratch_stride;
  // Problems in band_mask were given to the band kernel first; this kernel
  // solves them only where it fell back (band_fb[p] != 0).
  auto band_solved = [&](int p) { return ((band_mask >> p) & 1ull) && band_fb[p] == 0; };
  if (band_mask) {
    bool all = true;
    for (int p = 0; p < count && all; ++p) all = band_solved(p);
    if (all) return;
  }

  for (;;) {
    if (tid == 0) s_group = atomicAdd(counter, 1);
    __syncthreads();
    const int gg = s_group;
    if (gg >= total_groups) break;
    const GroupInfo gi = decode_group(tab, count, gg);
    const ProblemDev& pr = tab[gi.prob];
    if (band_mask && band_solved(gi.prob)) {
      // skip the rest of this problem's groups at once (the queue only grows)
      if (tid == 0) atomicMax(counter, pr.group_base + pr.num_groups);
      __syncthreads();
      continue;
    }
    if (pr.JT == kJTWide<T>) {
      solve_group<T, KMAX, kJTWide<T>>(pr, gi, sm, slice, sh.wide);
    } else if constexpr (kJTNarrow<T> != kJTWide<T>) {
      solve_group<T, KMAX, kJTNarrow<T>>(pr, gi, sm, slice, sh.narrow);
    }
  }
}

// C by quads of rows for the FP32 matvec: block b holds rows 4 b .. 4 b + 3 over
// the union of their columns in ascending order, entry e as the four rows'
// values qval[e][b] (zero where a row lacks the column) and the column's offset
// in the padded direction buffer qcol[e][b].  Neighbouring observations share
// most columns (a union is 1.05 to 1.3 times one row's count on 1-D and layered
// networks), so one 16-byte read of p and 20 bytes of C serve 16 FMAs; by rows
// it was a read of p and 8 bytes of C per 4.  One warp per block: the union as a bitmap
// in shared memory, a column's entry is its rank.  A union beyond the capacity sets
// status[2] and the matvec takes the rows.
constexpr int kQuadWarps = 4;
__global__ void __launch_bounds__(32 * kQuadWarps) k_pcg_quads(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.y];
  if (!pr.qval) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int JT = pr.JT, d = (int)pr.d, nb = (d + 3) / 4;
  const int blk = blockIdx.x * kQuadWarps + warp;
  if (blk >= nb) return;
  extern __shared__ uint32_t words_s[];   // per warp: bitmap, then the rank of each word's first bit
  const int nw = (d + 31) / 32;
  uint32_t* bits = words_s + (size_t)warp * 2 * nw;
  uint32_t* rank = bits + nw;
  for (int w = lane; w < nw; w += 32) bits[w] = 0;
  __syncwarp();
  const float* val = reinterpret_cast<const float*>(pr.oo_val);
#pragma unroll 1
  for (int i = 0; i < 4; ++i) {
    const int a = 4 * blk + i;
    const int nnz = a < d ? pr.oo_nnz[a] : 0;
    for (int e = lane; e < nnz; e += 32) {
      const int c = pr.oo_col[(int64_t)e * d + a];
      atomicOr(&bits[c >> 5], 1u << (c & 31));
    }
  }
  __syncwarp();
  int n = 0;
  for (int w0 = 0; w0 < nw; w0 += 32) {
    const int w = w0 + lane;
    const int cnt = w < nw ? __popc(bits[w]) : 0;
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    if (w < nw) rank[w] = (uint32_t)(n + incl - cnt);
    n += __shfl_sync(0xffffffffu, incl, 31);
  }
  __syncwarp();
  if (n > pr.qcap) {
    if (lane == 0) {
      pr.qn[blk] = 0;
      atomicExch(&pr.status[2], 1);
    }
    return;
  }
  if (lane == 0) pr.qn[blk] = n;
  float4* qv = reinterpret_cast<float4*>(pr.qval);
  for (int e = lane; e < n; e += 32) qv[(int64_t)e * nb + blk] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int w = lane; w < nw; w += 32) {
    uint32_t b = bits[w];
    int e = (int)rank[w];
    while (b) {
      const int c = 32 * w + __ffs(b) - 1;
      pr.qcol[(int64_t)e * nb + blk] = (int32_t)(p_row<float>(c) * JT);
      ++e;
      b &= b - 1;
    }
  }
  __syncwarp();   // the zeros before the values (same warp)
#pragma unroll 1
  for (int i = 0; i < 4; ++i) {
    const int a = 4 * blk + i;
    const int nnz = a < d ? pr.oo_nnz[a] : 0;
    for (int e = lane; e < nnz; e += 32) {
      const int c = pr.oo_col[(int64_t)e * d + a];
      const int at = (int)(rank[c >> 5] + __popc(bits[c >> 5] & ((1u << (c & 31)) - 1u)));
      pr.qval[((int64_t)at * nb + blk) * 4 + i] = val[(int64_t)e * d + a];
    }
  }
}

// Capacity of a problem's quads (0: none): FP32 problems that the general
// kernel solves, up to the size whose bitmaps fit and whose copy stays within
// 128 MB.
int64_t pcg_quad_cap(const ProblemDev& p, int count, int32_t solver, int32_t cluster_size) {
  if (p.precision != 1 || solver != 0 || p.d > 32768 || p.d < 1) return 0;
  const bool band = cluster_size > 0 || (cluster_size == 0 && count == 1);
  if (band && band1d_eligible(p)) return 0;
  const int64_t cap = std::min<int64_t>(p.d, 2 * p.max_oo + 8);
  return cap * ((p.d + 3) / 4) * 20 <= (int64_t(128) << 20) ? cap : 0;
}

void launch_pcg_quads(const ProblemTable& tab, const ProblemDev* dtab, cudaStream_t st) {
  int64_t dmax = 0;
  for (int i = 0; i < tab.count; ++i)
    if (tab.p[i].qval) dmax = std::max<int64_t>(dmax, tab.p[i].d);
  if (dmax < 1) return;
  const int smem = kQuadWarps * 2 * (int)((dmax + 31) / 32) * 4;   // 32 KB at most
  const unsigned nb = (unsigned)((dmax + 3) / 4);
  k_pcg_quads<<<dim3((nb + kQuadWarps - 1) / kQuadWarps, (unsigned)tab.count), 32 * kQuadWarps, smem, st>>>(dtab);
  note_launches(1);
}

// [Phi | C Phi] transposed, [2 k][d]: the columns that the kernel reads with
// consecutive rows on consecutive lanes.  Last step of the eigensolver's
// multi-kernel chain (the fused kernel writes it itself).
template <typename T>
__global__ void k_pcg_phit(const ProblemDev* tab) {
  const ProblemDev& pr = tab[blockIdx.y];
  const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int k = pr.kR;
  if (a >= pr.d || k <= 0) return;
  const T* P = reinterpret_cast<const T*>(pr.Phi);
  const T* A = reinterpret_cast<const T*>(pr.CPhi);
  T* out = reinterpret_cast<T*>(pr.phiT);
  for (int m = 0; m < k; ++m) {
    out[(int64_t)m * pr.d + a] = P[a * k + m];
    out[(int64_t)(k + m) * pr.d + a] = A[a * k + m];
  }
}

void launch_pcg_phit(const ProblemTable& tab, const ProblemDev* dtab, cudaStream_t st) {
  int64_t dmax = 1;
  for (int i = 0; i < tab.count; ++i) dmax = std::max<int64_t>(dmax, tab.p[i].d);
  const dim3 grid((unsigned)((dmax + 255) / 256), (unsigned)tab.count);
  if (tab.p[0].precision == 0) k_pcg_phit<double><<<grid, 256, 0, st>>>(dtab);
  else k_pcg_phit<float><<<grid, 256, 0, st>>>(dtab);
  note_launches(1);
}

// Systems per group of a problem with `systems` of them.  A CTA takes a group
// to its end, so the hardest group's iterations bound the call from below.
// FP64, whose pipe is the bound: groups of one halve that time where groups of
// two leave CTAs without work (100 weighted sums, 161 systems: 1.30 -> 1.12
// ms; at 321 systems, more groups of two than CTAs, 0.57 -> 0.61).  The line is
// where groups of two would have a CTA each.  One problem of 60 observations:
// groups of one take 0.53 ms from 141 to 241 systems and 0.58 at 301, groups of
// two 0.56 at 321; of 500 observations, 1.49 ms at 141 to 301 against 1.93 at 321.
// FP32: half a group's iteration costs almost what a whole one does (layered
// 961 systems 7.0 -> 7.3 ms).
// The rule looks at the problem alone, and so a batched call solves it in the
// same way, with the same bits, as a call of its own.  A batch that fills the chip
// anyway pays for that: 64 problems of 250 observations take 35.8 ms with 301
// systems each (groups of one) and 27.8 ms with 321.
int pcg_jt(int precision, int64_t systems, int num_sms) {
  if (precision != 0) return kJTWide<float>;
  return (systems + 1) / 2 <= num_sms ? kJTNarrow<double> : kJTWide<double>;
}

// Elements of one CTA's global slice: what the largest problem keeps there.
static size_t slice_elems(const ProblemTable& tab) {
  size_t most = 0;
  for (int i = 0; i < tab.count; ++i) {
    const bool f64 = tab.p[i].precision == 0;
    const PcgLayout l =
        f64 ? pcg_layout<double>(tab.p[i].d, tab.p[i].JT) : pcg_layout<float>(tab.p[i].d, tab.p[i].JT);
    const size_t need = l.level == 0 ? 0 : (l.level == 1 ? 3 * l.vec : 3 * l.vec + l.pvec);
    most = std::max(most, need);
  }
  return (most + 31) / 32 * 32;
}

size_t pcg_scratch_bytes(const ProblemTable& tab, int num_sms) {
  return slice_elems(tab) * (tab.p[0].precision == 0 ? 8 : 4) * (size_t)num_sms;   // one CTA per SM
}

// What a call must have of it.  The vectors of level 2 take 136 bytes a row in
// FP32 (with the padding of p); a call asks for no more than 128 bytes a row and SM,
// twice that up to rank 12, which is at least 16 CTAs of 17.  (BF16 only keeps
// directions here, see build_table.)
size_t pcg_scratch_least(const ProblemTable& tab, int num_sms) {
  const size_t full = pcg_scratch_bytes(tab, num_sms);
  const int precision = tab.p[0].precision;
  if (precision == 0) return full;
  int64_t dmax = 0, kmax = 0;
  for (int i = 0; i < tab.count; ++i) {
    dmax = std::max<int64_t>(dmax, tab.p[i].d);
    kmax = std::max<int64_t>(kmax, tab.p[i].kR);
  }
  const size_t slice = slice_elems(tab) * sizeof(float);
  const size_t room = (size_t)128 * dmax * num_sms * (precision == 1 && kmax <= 12 ? 2 : 1);
  return full <= room ? full : room / slice * slice;
}

template <typename T, int KMAX>
static int launch_pcg_t(const ProblemTable& tab, const ProblemDev* dtab, int32_t* counter, void* scratch,
                        size_t scratch_bytes, int num_sms, cudaStream_t st, uint64_t band_mask,
                        const int32_t* band_fb) {
  const size_t slice = slice_elems(tab);
  // the attribute once per thread and device
  constexpr int kMaxDev = 64;
  static thread_local bool attr_set[kMaxDev] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
    cudaGetLastError();
    dev = -1;
  }
  if (dev < 0 || !attr_set[dev]) {
    cudaFuncSetAttribute(k_pcg<T, KMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPcgSmem);
    if (dev >= 0) attr_set[dev] = true;
  }
  int64_t want = num_sms;
  if (slice > 0) want = std::min<int64_t>(want, (int64_t)(scratch_bytes / (slice * sizeof(T))));   // scratch slices
  const int grid = (int)std::min<int64_t>(tab.total_groups, want);
  if (grid < 1) return tab.total_groups > 0 ? -1 : 0;
  cudaMemsetAsync(counter, 0, sizeof(int32_t), st);
  k_pcg<T, KMAX><<<grid, kPcgThreads, kPcgSmem, st>>>(dtab, tab.count, tab.total_groups, counter,
                                                       reinterpret_cast<T*>(scratch), (int64_t)slice, band_mask,
                                                       band_fb);
  note_launches(1);
  return 0;
}

int launch_pcg(const ProblemTable& tab, const ProblemDev* dtab, int32_t* counter, void* scratch,
               size_t scratch_bytes, int num_sms, cudaStream_t st) {
  int kmax = 0;
  for (int i = 0; i < tab.count; ++i) kmax = tab.p[i].kR > kmax ? tab.p[i].kR : kmax;
  const bool small = kmax <= 12;
  // Problems the band kernel can take are launched there first, one launch
  // per problem (each with its own queue and fall-back flag in the counter
  // area); the general kernel then solves the rest and any that fell back.
  // cluster_size 0 uses the band kernel for a single problem only: in a batch
  // the general kernel packs the systems of many small problems onto all SMs
  // at once, while band launches run one after another, each with its own
  // drain (on 64 uneven problems the two came out within 2%, general first).
  const bool use_band = tab.cluster_size > 0 || (tab.cluster_size == 0 && tab.count == 1);
  int32_t* band_q = counter + 1;
  int32_t* band_fb = counter + 1 + kMaxProblems;
  uint64_t mask = 0;
  for (int i = 0; i < tab.count && use_band; ++i) {
    const ProblemDev& p = tab.p[i];
    if (!band1d_eligible(p)) continue;
    const int CS = band1d_cluster_size(p, tab.cluster_size);
    if (launch_pcg_band1d(p, dtab + i, CS, band_q + i, band_fb + i, num_sms, st) == 0) mask |= 1ull << i;
  }
  if (tab.p[0].precision == 0) {
    if (small) return launch_pcg_t<double, 12>(tab, dtab, counter, scratch, scratch_bytes, num_sms, st, mask, band_fb);
    return launch_pcg_t<double, 24>(tab, dtab, counter, scratch, scratch_bytes, num_sms, st, mask, band_fb);
  }
  if (small) return launch_pcg_t<float, 12>(tab, dtab, counter, scratch, scratch_bytes, num_sms, st, mask, band_fb);
  return launch_pcg_t<float, 24>(tab, dtab, counter, scratch, scratch_bytes, num_sms, st, mask, band_fb);
}

// ---------------------------------------------------------------------------
// Stage entry points for testing: Y = sigma P + C P and Z = P_q^-1 R for
// FP64 vectors [nvec][d] against the prepared band and Ritz pairs.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_obs_matvec(const ProblemDev* pr, int32_t nvec, const double* P, const double* sigma,
                             double* Y) {
  const int64_t d = pr->d;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= d * nvec) return;
  const int64_t v = i / d, a = i % d;
  const T* val = reinterpret_cast<const T*>(pr->oo_val);
  const T* Pv = nullptr;
  (void)Pv;
  T acc = to_t<T>(sigma[v]) * to_t<T>(P[v * d + a]);
  const int nnz = pr->oo_nnz[a];
  for (int e = 0; e < nnz; ++e)
    acc += val[(int64_t)e * d + a] * to_t<T>(P[v * d + pr->oo_col[(int64_t)e * d + a]]);
  Y[v * d + a] = (double)acc;
}

void launch_obs_matvec(const ProblemDev& pr, const ProblemDev* dpr, int32_t nvec, const double* P,
                       const double* sigma, double* Y, cudaStream_t st) {
  const int64_t tot = pr.d * nvec;
  if (tot <= 0) return;
  if (pr.precision == 0)
    k_obs_matvec<double><<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(dpr, nvec, P, sigma, Y);
  else
    k_obs_matvec<float><<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(dpr, nvec, P, sigma, Y);
  note_launches(1);
}

// One block per vector; same algebra as the PCG kernel, FP64 throughout.
template <typename T>
__global__ void k_lmp_apply(const ProblemDev* prp, int32_t nvec, const double* Rv, const double* sigma_in,
                            double* Z) {
  const ProblemDev& pr = *prp;
  const int64_t d = pr.d;
  const int k = pr.kR;
  const int v = blockIdx.x;
  const double* r = Rv + (int64_t)v * d;
  double* z = Z + (int64_t)v * d;
  const double sigma = sigma_in[v];
  const T* Phi = reinterpret_cast<const T*>(pr.Phi);
  const T* A = reinterpret_cast<const T*>(pr.CPhi);
  __shared__ double fg[2 * kMaxK][kThreads / 32];
  __shared__ double cc[2][kMaxK];
  for (int m = 0; m < 2 * k; ++m) {
    double acc = 0.0;
    for (int64_t a = threadIdx.x; a < d; a += blockDim.x)
      acc += (double)(m < k ? Phi[a * k + m] : A[a * k + (m - k)]) * r[a];
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) fg[m][threadIdx.x >> 5] = acc;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double f[kMaxK], g[kMaxK], t[kMaxK];
    for (int m = 0; m < 2 * k; ++m) {
      double s = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += fg[m][w];
      if (m < k) f[m] = s; else g[m - k] = s;
    }
    const double beta = sigma + pr.scal[1];
    for (int m = 0; m < k; ++m) t[m] = f[m] / (pr.theta[m] + sigma);
    for (int m = 0; m < k; ++m) {
      double t2 = g[m] + sigma * f[m];
      for (int i = 0; i < k; ++i) {
        const int e = m * k + i;
        const double G = pr.gram[2 * k * k + e] + sigma * (pr.gram[k * k + e] + pr.gram[k * k + i * k + m]) +
                         sigma * sigma * pr.gram[e];
        t2 -= G * t[i];
      }
      cc[0][m] = t[m];
      cc[1][m] = (beta - sigma) * t[m] - t2 / (pr.theta[m] + sigma);
    }
  }
  __syncthreads();
  for (int64_t a = threadIdx.x; a < d; a += blockDim.x) {
    double acc = r[a];
    for (int m = 0; m < k; ++m) acc += (double)Phi[a * k + m] * cc[1][m] - (double)A[a * k + m] * cc[0][m];
    z[a] = acc;
  }
}

void launch_lmp_apply(const ProblemDev& pr, const ProblemDev* dpr, int32_t nvec, const double* Rv,
                      const double* sigma, double* Z, cudaStream_t st) {
  if (nvec <= 0) return;
  if (pr.precision == 0) k_lmp_apply<double><<<nvec, kThreads, 0, st>>>(dpr, nvec, Rv, sigma, Z);
  else k_lmp_apply<float><<<nvec, kThreads, 0, st>>>(dpr, nvec, Rv, sigma, Z);
  note_launches(1);
}

}  // namespace infoesrf
