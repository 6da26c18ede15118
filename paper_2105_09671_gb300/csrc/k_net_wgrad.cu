// Weight and bias gradients of the jump network's 32 -> 32 layers on the
// tensor cores:
//
//   dW[t][ci][co] += sum_p a[p + t][ci] * g[p][co],   db[co] += sum_p g[p][co]
//
// The reduction runs over the pixels, which are the slow index of both
// operands in memory: both are fed to the MMA as they lie (MN-major operands:
// channels contiguous, pixels strided), so staging is TMA copies only.
//
// Work item: two rows of g by 128 pixels (one z, one image) and the four
// padded rows of a that the taps of one dz reach from them.  A stage holds 4
// rows x 130 pixels of a and 2 rows x 128 pixels of g, 64 bytes (32 channels)
// a pixel in the 64-byte swizzle, one TMA box each:
//   A = a: M = 128 = (a row 0..3, channel), K = 16 pixels,
//   B = g: N = 64 = (g row 0..1, channel),
// and the x offset of a tap is +64 bytes on A's start address, so a stage is
// 3 (ox) x 8 (k) MMAs into 3 TMEM accumulators that live for the whole CTA.
// Of the 4 x 2 (a row, g row) pairs 6 are taps (oy = a row - g row - 1), the
// other two are dropped.  In 3D blockIdx.y is the tap's dz.
//
// Bound: reading A from shared memory (4 KB per MMA at 128 B a clock, 32 of
// ~48 clocks) and the L2 reads (192 bytes a pixel, a rows twice).  The kernel
// before this one built the operands with 2-byte shared-memory stores by all
// threads, one chunk at a time, waiting for each MMA: 32 x 256^2 pixels took
// 2809 us a layer, this one 72 (272 MB from DRAM: 40 us at the copy rate).
//
// Warp 0 issues the TMA loads, warp 1 the MMAs, warps 2 and 3 sum g for the
// bias; all four add the accumulators to the global gradient at the end.
// Every wait is bounded; on expiry the status word is set and the roles wind
// down without leaving copies or MMAs in flight.
#include "kernels.h"
#include "net.cuh"
#include "tc.cuh"

namespace ac {

namespace {

constexpr int kWgPix = 128;                         // pixels of g per row of an item
constexpr int kWgRowA = (kWgPix + 2) * 64;          // bytes: one row of a
constexpr int kWgRowG = kWgPix * 64;                // one row of g
constexpr int kWgStageG = 4 * kWgRowA;              // offset of g in a stage
constexpr int kWgStage = 4 * kWgRowA + 2 * kWgRowG;
constexpr int kWgStages = 4;
constexpr int kWgThreads = 128;
constexpr int kWgTmem = 256;                        // 3 accumulators of 64 columns
constexpr int kWgSmem = kWgStages * kWgStage + (2 * kWgStages + 1) * 8 + 8;
static_assert(kWgStageG % 512 == 0 && kWgStage % 512 == 0, "the swizzle pattern repeats every 512 bytes");
static_assert(kWgSmem <= 227 * 1024, "shared memory");

// kind::f16, BF16 x BF16 -> FP32, M = 128, N = 64, both operands MN-major
// (transpose bits 15 and 16).
constexpr uint32_t kWgIdesc = tc_idesc_bf16_f32(128, 64) | (1u << 15) | (1u << 16);

struct WgItem {
  int b, z, y, x0;
};
__device__ __forceinline__ WgItem wg_item(int64_t i, const NetShape &sh, int tiles_x, int pairs) {
  WgItem it;
  it.x0 = (int)(i % tiles_x) * kWgPix;
  i /= tiles_x;
  it.y = (int)(i % pairs) * 2;
  i /= pairs;
  it.z = (int)(i % sh.nz);
  it.b = (int)(i / sh.nz);
  return it;
}

}  // namespace

template <int NDIM>
__global__ void __launch_bounds__(kWgThreads, 1)
    net_wgrad_rows_k(const __grid_constant__ CUtensorMap a_map, const __grid_constant__ CUtensorMap g_map,
                     NetShape sh, float *__restrict__ gw, float *__restrict__ gb, int *status) {
  extern __shared__ __align__(1024) unsigned char sm[];
  uint64_t *full = reinterpret_cast<uint64_t *>(sm + kWgStages * kWgStage);
  uint64_t *empty = full + kWgStages;
  uint64_t *fin = empty + kWgStages;
  uint32_t *tslot = reinterpret_cast<uint32_t *>(fin + 1);
  volatile int &abort_flag = *reinterpret_cast<volatile int *>(tslot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int dz = NDIM == 3 ? blockIdx.y : 0;
  if (tid == 0) {
    tma_prefetch_desc(&a_map);
    tma_prefetch_desc(&g_map);
    for (int s = 0; s < kWgStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 3);  // the MMAs' commit and the two bias warps
    }
    mbar_init(fin, 1);
    fence_mbar_init();
    abort_flag = 0;
  }
  if (warp == 1) {
    tmem_alloc(tslot, kWgTmem);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  const int tiles_x = (sh.nx + kWgPix - 1) / kWgPix, pairs = (sh.ny + 1) / 2;
  const int64_t items = (int64_t)sh.batch * sh.nz * pairs * tiles_x;
  const bool any = blockIdx.x < items;
  float bias[32];

  if (warp == 0) {
    if (lane == 0) {
      uint32_t i = 0;  // stages filled
      bool ok = true;
      for (int64_t item = blockIdx.x; item < items; item += gridDim.x, ++i) {
        const int s = (int)(i % kWgStages);
        if (i >= (uint32_t)kWgStages) ok = mbar_wait_bounded(&empty[s], (i / kWgStages - 1) & 1u);
        if (!ok || abort_flag) { ok = false; break; }
        const WgItem it = wg_item(item, sh, tiles_x, pairs);
        unsigned char *st = sm + s * kWgStage;
        mbar_arrive_expect_tx(&full[s], kWgStage);
        // rows of the padded arrays; columns and rows past the end are filled
        // with zeros, and g's ghost ring is zero (the second row of an odd ny)
        const int64_t row0 = ((int64_t)it.b * sh.pz()) * sh.py() + it.y;
        const int ra = (int)(row0 + (NDIM == 3 ? (int64_t)(it.z + dz) * sh.py() : 0));
        const int rg = (int)(row0 + 1 + (NDIM == 3 ? (int64_t)(it.z + 1) * sh.py() : 0));
        tma_load_3d(st, &a_map, &full[s], 0, it.x0, ra);
        tma_load_3d(st + kWgStageG, &g_map, &full[s], 0, it.x0 + 1, rg);
      }
      if (!ok && !abort_flag) {
        report_timeout(status);
        abort_flag = 1;
      }
      // never leave with a copy in flight
      for (uint32_t v = i > (uint32_t)kWgStages ? i - kWgStages : 0; v < i; ++v)
        mbar_wait_bounded(&full[v % kWgStages], (v / kWgStages) & 1u);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      uint32_t i = 0;
      bool ok = true;
      for (int64_t item = blockIdx.x; item < items; item += gridDim.x, ++i) {
        const int s = (int)(i % kWgStages);
        ok = mbar_wait_bounded(&full[s], (i / kWgStages) & 1u);
        if (!ok || abort_flag) { ok = false; break; }
        tc_fence_after();
        unsigned char *st = sm + s * kWgStage;
        // MN-major in the 64-byte swizzle: LBO between blocks of 32 channels
        // (rows), SBO between groups of 8 pixels
        const uint64_t da = tc_smem_desc_sw64(st, kWgRowA, 512);
        const uint64_t db = tc_smem_desc_sw64(st + kWgStageG, kWgRowG, 512);
#pragma unroll
        for (int kk = 0; kk < kWgPix / 16; ++kk)
#pragma unroll
          for (int ox = 0; ox < 3; ++ox)
            tc_mma_bf16(tmem + ox * 64, da + (uint32_t)((kk * 1024 + ox * 64) >> 4),
                        db + (uint32_t)((kk * 1024) >> 4), kWgIdesc, i > 0 || kk > 0);
        tc_commit(&empty[s]);
      }
      if (!ok && !abort_flag) {
        report_timeout(status);
        abort_flag = 1;
      }
      tc_commit(fin);  // every MMA issued has completed before TMEM is read or freed
    }
  } else {
    // bias: this warp's g row of every item (dz = the middle plane in 3D)
#pragma unroll
    for (int c = 0; c < 32; ++c) bias[c] = 0.f;
    const bool sums = NDIM == 2 || dz == 1;
    uint32_t i = 0;
    for (int64_t item = blockIdx.x; item < items; item += gridDim.x, ++i) {
      const int s = (int)(i % kWgStages);
      const bool ok = mbar_wait_bounded(&full[s], (i / kWgStages) & 1u) && !abort_flag;
      if (!__all_sync(0xffffffffu, ok)) {
        if (lane == 0 && !abort_flag) {
          report_timeout(status);
          abort_flag = 1;
        }
        break;
      }
      if (sums) {
        const unsigned char *gr = sm + s * kWgStage + kWgStageG + (warp - 2) * kWgRowG + lane * 64;
        const int sw = (lane >> 1) & 3;  // the swizzle of this lane's pixels
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int m = 0; m < kWgPix / 32; ++m) {
            float v[8];
            unpack8_bf16(*reinterpret_cast<const uint4 *>(gr + m * 2048 + ((c ^ sw) << 4)), v);
#pragma unroll
            for (int e = 0; e < 8; ++e) bias[c * 8 + e] += v[e];
          }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[s]);
    }
    if (any && sums) {
      // lane c keeps channel c's total of the warp
      float mine = 0.f;
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        float v = bias[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == c) mine = v;
      }
      atomicAdd(gb + lane, mine);
    }
  }
  __syncwarp();
  const bool done = mbar_wait_bounded(fin, 0);
  if (!done && tid == 0) report_timeout(status);
  __syncwarp();
  tc_fence_after();
  if (any && done) {
    // accumulator lane: a row = warp, channel = lane; column: g row, channel
#pragma unroll
    for (int ox = 0; ox < 3; ++ox)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int oy = warp - h;
        if (oy < 0 || oy > 2) continue;
        float v[32];
        tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + ox * 64 + h * 32, v);
        float4 *d = reinterpret_cast<float4 *>(gw + ((int64_t)(dz * 9 + oy * 3 + ox) * kNetC + lane) * kNetC);
#pragma unroll
        for (int q = 0; q < 8; ++q)
          atomicAdd(d + q, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
      }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, kWgTmem);
}

// ------------------------------------------------------------------ host ---
template <int NDIM>
static cudaError_t wgrad_t(const bf16 *apad, const bf16 *gpad, const NetShape &sh, float *gw, float *gb,
                           int *status, int num_sms, cudaStream_t s) {
  static KernelSetup ks;
  int occ = 1;
  cudaError_t e = kernel_setup(ks, (const void *)net_wgrad_rows_k<NDIM>, kWgThreads, kWgSmem, &occ);
  if (e != cudaSuccess) return e;
  EncodeTiledFn fn = ac_encode_fn();
  if (!fn) return cudaErrorNotSupported;
  // padded arrays as {32 channels, padded columns, rows of all planes and images}
  const int64_t rows = (int64_t)sh.batch * sh.pz() * sh.py();
  if (rows + 4 >= (int64_t)INT32_MAX) return cudaErrorInvalidValue;
  const cuuint64_t dims[3] = {(cuuint64_t)kNetC, (cuuint64_t)sh.px(), (cuuint64_t)rows};
  const cuuint64_t strides[2] = {(cuuint64_t)kNetC * 2, (cuuint64_t)sh.px() * kNetC * 2};
  const cuuint32_t es[3] = {1, 1, 1};
  CUtensorMap maps[2];
  for (int w = 0; w < 2; ++w) {
    const cuuint32_t box[3] = {(cuuint32_t)kNetC, (cuuint32_t)(w ? kWgPix : kWgPix + 2), (cuuint32_t)(w ? 2 : 4)};
    if (fn(&maps[w], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16 *>(w ? gpad : apad), dims, strides,
           box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  const int64_t items = (int64_t)sh.batch * sh.nz * ((sh.ny + 1) / 2) * ((sh.nx + kWgPix - 1) / kWgPix);
  const int planes = NDIM == 3 ? 3 : 1;
  const dim3 grid((unsigned)std::min<int64_t>(items, std::max(1, num_sms / planes)), planes);
  net_wgrad_rows_k<NDIM><<<grid, kWgThreads, kWgSmem, s>>>(maps[0], maps[1], sh, gw, gb, status);
  return cudaGetLastError();
}

cudaError_t net_wgrad(const bf16 *apad, const bf16 *gpad, const NetShape &sh, float *gw, float *gb, int *status,
                      int num_sms, cudaStream_t s) {
  return sh.ndim == 3 ? wgrad_t<3>(apad, gpad, sh, gw, gb, status, num_sms, s)
                      : wgrad_t<2>(apad, gpad, sh, gw, gb, status, num_sms, s);
}

}  // namespace ac
