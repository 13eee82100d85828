// a5, BF16 path: the localized-covariance matvec of every PCG iteration,
//     y_j = sigma_j p_j + C p_j   for all systems j at once
// (App. E, Eq. normalized_linear_solve; every shifted system shares the one
// matrix C = R^-1/2 (L_oo o W W^T) R^-1/2 of Sec. 2.3, so the product over
// all systems is one block-sparse matrix product C P with P = [p_1 ... p_J]).
//
// Layout.  Observations are numbered in tile order (the library's own
// permutation, spatially compact tiles).  C is kept only in the 128 x 64
// blocks (row tile, column block) whose bounding boxes come within the
// Gaspari-Cohn support (all other entries are exact zeros), each block
// stored as two BF16 planes hi = bf16(C), lo = bf16(C - hi), row-major
// [tile][128][64].  The directions are BF16, system-major [J][d_pad].
//
// Kernel.  The running systems' directions are consecutive rows of P (the PCG
// keeps them by position), so a launch covers ceil(count / 16) units of 16
// rows, split evenly over `nchunks` CTAs per row tile (at most BN / 16 units
// each): converged systems cost no tensor-core work.  One CTA of 4 warps per
// (row tile, chunk): warp 0 lane 0 streams the blocks of the row tile through
// an S-stage ring of shared memory with 2-D TMA loads (128-byte swizzle): the
// hi and lo planes of the C block (the A operand, 128 x 64, K-major) and one
// slab of directions (the B operand, 16 u x 64, K-major).  The row tile's
// column-block list is staged in shared memory first: read from global memory
// inside the loop, its latency stood in front of every stage's loads.  Warp 1
// lane 0 issues tcgen05.mma kind::f16 (BF16 x BF16, FP32 accumulate, N = 16 u)
// into a 128 x 16 u FP32 accumulator in tensor memory: four K = 16 steps for
// hi, four for lo, then a commit that frees the stage.  After the last block
// all four warps read the accumulator (tcgen05.ld, one TMEM lane = one row per
// thread), add sigma_j p_j, store y and reduce the partial dot products
// p_j^T y_j of the row tile.
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include "common.cuh"
#include "info_esrf_stages.h"
#include "internal.h"
#include "tile_mma.cuh"

namespace infoesrf {

namespace {

constexpr int kABytes = kTileM * kTileK * 2;     // one BF16 plane of a C block: 16 KB
constexpr int kUnitBytes = kTileUnit * kTileK * 2;   // one unit's slab of P: 2 KB

constexpr int kMaxList = 1024;                       // column blocks of a row tile staged in shared memory

// At most BN systems (BN / 16 units) per CTA, S pipeline stages.
template <int BN, int S>
struct TileMmShape {
  static constexpr int kUnits = BN / kTileUnit;
  static constexpr int kStage = 2 * kABytes + BN * kTileK * 2;
  static constexpr int kCtrl = 128;   // mbarriers, TMEM slot, flags
  static_assert(8 * (2 * S + 1) + 4 + 12 <= kCtrl, "control block");
  static constexpr size_t kSmem = 1024 + (size_t)S * kStage + kCtrl + kMaxList * 4 + 5 * BN * sizeof(float);
};

template <int BN, int S>
__global__ void __launch_bounds__(128, 1)
    k_tile_mm(const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo,
              const __grid_constant__ CUtensorMap map_p, const TileMmArgs args) {
  using Shape = TileMmShape<BN, S>;
  constexpr int kStage = Shape::kStage;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                         ~static_cast<uintptr_t>(1023));
  unsigned char* ctrl = smem + S * kStage;
  uint64_t* full = reinterpret_cast<uint64_t*>(ctrl);
  uint64_t* empty = full + S;
  uint64_t* accf = empty + S;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(accf + 1);
  int* flags = reinterpret_cast<int*>(tslot + 1);   // [0] abort, [1] loads issued, [2] stages consumed
  int* cols = reinterpret_cast<int*>(ctrl + Shape::kCtrl);   // the row tile's column blocks (the first kMaxList)
  float* red = reinterpret_cast<float*>(cols + kMaxList);
  float* sg = red + 4 * BN;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  grid_dependency_wait();
  // an overflowed block pattern is not read (uniform across the grid)
  if (args.status && (*reinterpret_cast<volatile int32_t*>(args.status) & kStatTileOverflow)) return;
  const int chunk = (int)(blockIdx.x % (unsigned)args.nchunks);
  const int rt = (int)(blockIdx.x / (unsigned)args.nchunks);
  // this CTA's rows of P: [c0, c0 + ncol), ncol a multiple of 16
  const int T = args.count ? *args.count : args.J;
  const int c0 = chunk * args.upc * kTileUnit;
  if (c0 >= T) return;   // uniform across the CTA, before any barrier or TMEM use
  const int nu = min(args.upc, (T - c0 + kTileUnit - 1) / kTileUnit);
  const int ncol = nu * kTileUnit;
  const uint32_t stage_bytes = 2 * kABytes + args.upc * kUnitBytes;
  const int t0 = args.rowptr[rt];
  const int nk = args.rowptr[rt + 1] - t0;
  for (int e = threadIdx.x; e < min(nk, kMaxList); e += 128) cols[e] = args.colblk[t0 + e];
  for (int t = threadIdx.x; t < ncol; t += 128) {   // the columns' shifts
    const int j = c0 + t;
    sg[t] = j < T && args.sigma ? args.sigma[args.list ? args.list[j] : j] : 0.f;
  }

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accf, 1);
    flags[0] = 0;
    flags[1] = 0;
    flags[2] = 0;
    fence_mbar_init();
    tma_prefetch_map(&map_hi);
    tma_prefetch_map(&map_lo);
    tma_prefetch_map(&map_p);
  }
  if (warp == 2) tmem_alloc(tslot, BN);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  if (warp == 0 && lane == 0) {
    // producer: C block planes and each unit's slab of the directions for the block's columns
    int kb = 0;
    for (; kb < nk; ++kb) {
      const int s = kb % S;
      if (kb >= S && !mbar_wait(&empty[s], ((kb / S) & 1) ^ 1)) {
        atomicExch(&flags[0], 1);
        break;
      }
      if (*reinterpret_cast<volatile int*>(&flags[0])) break;
      unsigned char* st = smem + s * kStage;
      const int tile = t0 + kb;
      const int xcol = (kb < kMaxList ? cols[kb] : args.colblk[tile]) * kTileK;
      mbar_arrive_expect_tx(&full[s], stage_bytes);
      tma_load_2d(st, &map_hi, &full[s], 0, tile * kTileM);
      tma_load_2d(st + kABytes, &map_lo, &full[s], 0, tile * kTileM);
      tma_load_2d(st + 2 * kABytes, &map_p, &full[s], xcol, c0);
    }
    flags[1] = kb;
  } else if (warp == 1 && lane == 0) {
    // MMA issuer: acc = sum over blocks of (C_hi + C_lo) P, FP32 in TMEM
    const uint32_t idesc = idesc_bf16_f32(kTileM, ncol);
    int kb = 0;
    for (; kb < nk; ++kb) {
      const int s = kb % S;
      if (!mbar_wait(&full[s], (kb / S) & 1)) {
        atomicExch(&flags[0], 1);
        break;
      }
      tc_fence_after();
      const uint32_t base = smem_u32(smem + s * kStage);
      const uint64_t dhi = sw128_desc(base), dlo = sw128_desc(base + kABytes);
      const uint64_t db = sw128_desc(base + 2 * kABytes);
#pragma unroll
      for (int k = 0; k < kTileK / 16; ++k)   // K = 16 per MMA: 32 bytes along the swizzled row
        mma_bf16(tmem, dhi + 2 * k, db + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
#pragma unroll
      for (int k = 0; k < kTileK / 16; ++k) mma_bf16(tmem, dlo + 2 * k, db + 2 * k, idesc, 1u);
      mma_commit(&empty[s]);
    }
    flags[2] = kb;
    mma_commit(accf);
  }
  __syncwarp();
  if (!mbar_wait(accf, 0)) atomicExch(&flags[0], 1);
  tc_fence_after();
  __syncthreads();
  const bool aborted = *reinterpret_cast<volatile int*>(&flags[0]) != 0;
  if (!aborted) {
    const int row = warp * 32 + lane;
    const int64_t a = (int64_t)rt * kTileM + row;
    const uint32_t tbase = tmem + ((uint32_t)(warp * 32) << 16);
    // One unit = 16 accumulator columns.  Every load of a unit is issued before
    // its first use and the next unit's p under the current one: with a column at
    // a time, the stores of y kept the loads of the next column behind them (three
    // dependent reads a column: 66 us a launch at 15 row tiles x 961 systems, 30 us
    // now, and 252 -> 211 ms for an analysis of 512 x 512 points).
    auto load_p = [&](float (&p)[kTileUnit], int i) {
      const __nv_bfloat16* src = args.P + (int64_t)(c0 + i * kTileUnit) * args.d_pad + a;
#pragma unroll
      for (int c = 0; c < kTileUnit; ++c)
        p[c] = c0 + i * kTileUnit + c < T ? __bfloat162float(src[(int64_t)c * args.d_pad]) : 0.f;
    };
    float p[kTileUnit];
    load_p(p, 0);
    for (int i = 0; i < nu; ++i) {
      float v[kTileUnit], pn[kTileUnit];
      tmem_ld16(tbase + (uint32_t)(i * kTileUnit), v);
      if (i + 1 < nu) load_p(pn, i + 1);
      const int jb = c0 + i * kTileUnit;
      float* dst = args.Y + (int64_t)jb * args.d_pad + a;
#pragma unroll
      for (int c = 0; c < kTileUnit; ++c) {
        const float y = fmaf(sg[i * kTileUnit + c], p[c], v[c]);
        if (jb + c < T) dst[(int64_t)c * args.d_pad] = y;
        v[c] = p[c] * y;   // p = 0 past the last system
      }
      // sums over the warp's rows: halve the columns a lane holds, then the lane pairs
      // (the same tree as a butterfly per column)
      int idx = 0;
#pragma unroll
      for (int off = 16, w = kTileUnit / 2; w >= 1; off >>= 1, w >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int c = 0; c < w; ++c) {
          const float send = up ? v[c] : v[c + w];
          const float keep = up ? v[c + w] : v[c];
          v[c] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
        if (up) idx += w;
      }
      const float dot = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
      if ((lane & 1) == 0) red[warp * BN + i * kTileUnit + idx] = dot;
#pragma unroll
      for (int c = 0; c < kTileUnit; ++c) p[c] = pn[c];
    }
    __syncthreads();
    if (args.pty)
      for (int t = threadIdx.x; t < ncol; t += blockDim.x) {
        const int j = c0 + t;
        if (j < T) {
          const float v = (red[t] + red[BN + t]) + (red[2 * BN + t] + red[3 * BN + t]);
          if (args.pty_by_system) args.pty[(int64_t)j * args.nrt + rt] = v;
          else args.pty[(int64_t)rt * args.J + j] = v;
        }
      }
  } else if (threadIdx.x == 0) {
    // wait (bounded) for the loads still in flight before the CTA's shared memory goes away
    for (int kb = flags[2]; kb < flags[1]; ++kb) mbar_wait(&full[kb % S], (kb / S) & 1);
    if (args.status) atomicOr(args.status, kStatTimeout);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) tmem_dealloc(tmem, BN);
}

template <int BN, int S>
int launch_tile_mm_t(TileMmArgs a, int units, const void* chi, const void* clo, int64_t ntiles, cudaStream_t st) {
  using Shape = TileMmShape<BN, S>;
  a.nchunks = (units + Shape::kUnits - 1) / Shape::kUnits;
  a.upc = (units + a.nchunks - 1) / a.nchunks;
  CUtensorMap mh, ml, mp;
  if (!encode_bf16(&mh, chi, kTileK, (uint64_t)ntiles * kTileM, kTileK, kTileM) ||
      !encode_bf16(&ml, clo, kTileK, (uint64_t)ntiles * kTileM, kTileK, kTileM) ||
      !encode_bf16(&mp, a.P, (uint64_t)a.d_pad, (uint64_t)a.J, (uint64_t)a.d_pad, (uint32_t)(kTileUnit * a.upc)))
    return INFO_ESRF_ERR_CUDA;
  static thread_local int raised_dev = -1;
  int dev = 0;
  cudaGetDevice(&dev);
  if (raised_dev != dev) {
    if (cudaFuncSetAttribute(k_tile_mm<BN, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Shape::kSmem) !=
        cudaSuccess)
      return INFO_ESRF_ERR_CUDA;
    raised_dev = dev;
  }
  const int64_t grid = (int64_t)a.nrt * a.nchunks;
  launch_overlapped(k_tile_mm<BN, S>, dim3((unsigned)grid), 128, Shape::kSmem, st, mh, ml, mp, a);
  note_launches(1);
  return cudaGetLastError() == cudaSuccess ? INFO_ESRF_OK : INFO_ESRF_ERR_CUDA;
}

}  // namespace

int launch_tile_mm(TileMmArgs a, const void* chi, const void* clo, int64_t ntiles, cudaStream_t st) {
  if (a.nrt < 1 || a.J < 1 || a.d_pad % kTileM || (int64_t)a.nrt * kTileM != a.d_pad ||
      ntiles * kTileM >= (int64_t(1) << 31) || (a.count && (a.J_run < 0 || a.J_run > a.J)))
    return INFO_ESRF_ERR_INVALID_ARG;
  const int units = ((a.count ? a.J_run : a.J) + kTileUnit - 1) / kTileUnit;
  if (units == 0) return INFO_ESRF_OK;
  // up to 4 units (64 systems): 5 stages of 40 KB; up to 8 units: a 128-column
  // accumulator and 4 stages; else up to 16 units per CTA, 3 stages.  (Two
  // 256-column accumulators per CTA, so that a C block load serves 512
  // systems, leave room for two stages only and measured slower: 1225 against
  // 1273 TFLOP/s on the tilemm workload.)
  if (units <= 4) return launch_tile_mm_t<64, 5>(a, units, chi, clo, ntiles, st);
  if (units <= 8) return launch_tile_mm_t<128, 4>(a, units, chi, clo, ntiles, st);
  return launch_tile_mm_t<256, 3>(a, units, chi, clo, ntiles, st);
}

}  // namespace infoesrf

using namespace infoesrf;

extern "C" int info_esrf_bf16_tile_matvec(int32_t n_row_tiles, const int32_t* rowptr_dev, const int32_t* colblk_dev,
                                          int64_t n_tiles, const uint16_t* C_hi_dev, const uint16_t* C_lo_dev,
                                          int32_t J, const uint16_t* P_dev, const float* sigma_dev, float* Y_dev,
                                          float* pty_dev, int32_t* status_dev, void* stream) {
  if (n_row_tiles < 1 || n_tiles < n_row_tiles || J < 1 || !rowptr_dev || !colblk_dev || !C_hi_dev || !C_lo_dev ||
      !P_dev || !sigma_dev || !Y_dev)
    return INFO_ESRF_ERR_INVALID_ARG;
  TileMmArgs a{};
  a.rowptr = rowptr_dev;
  a.colblk = colblk_dev;
  a.P = reinterpret_cast<const __nv_bfloat16*>(P_dev);
  a.sigma = sigma_dev;
  a.Y = Y_dev;
  a.pty = pty_dev;
  a.status = status_dev;
  a.d_pad = (int64_t)n_row_tiles * kTileM;
  a.J = J;
  a.nrt = n_row_tiles;
  cudaGetLastError();
  return launch_tile_mm(a, C_hi_dev, C_lo_dev, n_tiles, reinterpret_cast<cudaStream_t>(stream));
}

namespace infoesrf {
namespace {

// One bounded mbarrier wait, as the tensor-core kernels wait for their copies
// and MMAs: thread 0 initializes a barrier of one arrival, arrives on it first
// when `arrive` is set, then waits for its phase 0 at most `limit` cycles and
// records kStatTimeout in *status when the wait ran out.  Nothing faults or
// hangs: with no arrival the wait ends after the limit.
__global__ void k_wait_probe(long long limit, int arrive, int32_t* status) {
  __shared__ uint64_t bar;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);
  fence_mbar_init();
  if (arrive) mbar_arrive(&bar);
  status[0] = mbar_wait(&bar, 0, limit) ? 0 : kStatTimeout;
}

}  // namespace
}  // namespace infoesrf

extern "C" int info_esrf_wait_probe(int64_t limit_cycles, int32_t arrive, int32_t* status_dev, void* stream) {
  if (!status_dev || limit_cycles < 1 || limit_cycles > infoesrf::kWaitCycles) return INFO_ESRF_ERR_INVALID_ARG;
  cudaGetLastError();
  infoesrf::k_wait_probe<<<1, 32, 0, reinterpret_cast<cudaStream_t>(stream)>>>((long long)limit_cycles,
                                                                                arrive ? 1 : 0, status_dev);
  infoesrf::note_launches(1);
  return cudaGetLastError() == cudaSuccess ? INFO_ESRF_OK : INFO_ESRF_ERR_CUDA;
}
