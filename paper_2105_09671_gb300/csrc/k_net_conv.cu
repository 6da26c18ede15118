// Row-streaming tensor-core convolution of the jump network (the 32 -> 32
// layers, forward and data gradient):
//
//   out[p][n] = sum_{t < T} sum_{c < 32} in[p + t][c] * Wx[n][t*32 + c]
//
// Work item: 128 consecutive x positions of a run of output rows (one z, one
// image).  Each input row reaches shared memory once, by TMA, and is used
// once, for the three output rows that it touches:
//   - one padded input row is the 130 pixels x0-1 .. x0+128 at 64 bytes (32
//     channels) each, one 2D TMA box in the 64-byte swizzle (K-major), so an x
//     offset of a tap is +64 bytes on the descriptor's start address and the
//     second half of the channels +32;
//   - warp 0 (one thread) issues the TMA loads into a ring of row sets (the
//     1 or 3 rows of one y at every needed z), each set on a full / empty
//     mbarrier pair;
//   - TMEM holds a ring of 8 output rows of 32 columns.  Input row r adds to
//     output rows r-1, r, r+1 (through the taps oy = +1, 0, -1), which are
//     adjacent blocks of columns: with the weights of the three oy side by
//     side in N, one tcgen05.mma (M = 128 pixels, N = 96, K = 16) per ox, dz
//     and half of the channels serves all three.  The MMA that touches an
//     output row first starts it from zero (N = 32), and a triple that wraps
//     around the ring is split in two.  Warp 1 (one thread) issues them (its
//     own latency counts: operands that cost ~50 instructions an MMA to form
//     made a row take 2200 clocks) and
//     commits to the set's empty barrier and, once its last tap is in, to the
//     output row's barrier;
//   - warps 2..9 read finished rows (tcgen05.ld, lanes 32 (w % 4) ..; two
//     groups of four warps take alternate rows), release them, and run the
//     epilogue: bias, pre-activation store, GELU (tanh form, hardware tanh
//     approximation) and the store with its replicated ghost ring; or, for the
//     data gradient, x gelu'(z) and the store into the padded gradient for
//     cells inside the grid, the raw FP32 sum for cells on its faces
//     (net_dgrad_faces adds what their ghosts received).
// Bound: operand reads from shared memory.  With one MMA per tap (N = 32) the
// A rows were read 18 times (2D) instead of 6 to 8 times: 720 clocks of
// 128-byte reads per 128-pixel row.  In training the activations come next:
// 32 x 256^2 pixels move 400 MB a layer (59 us at the copy rate) and take 80 us
// forward, 87 us for the data gradient; 1024^2 without pre-activations 33 us
// (47 before the three rows shared an MMA).  A third epilogue group: 86 us.
// Every wait is bounded; a timeout sets the status word and the roles wind
// down without leaving copies or MMAs in flight.
#include "kernels.h"
#include "net.cuh"
#include "tc.cuh"

namespace ac {

namespace {

constexpr int kCvPix = 130;                // 128 outputs + 2 halo columns
constexpr int kCvBox = kCvPix * 64;        // bytes of one input row (one TMA box)
constexpr int kCvRow = (kCvBox + 511) / 512 * 512;  // its place (the swizzle pattern repeats every 512)
constexpr int kCvThreads = 320;  // TMA warp, MMA warp, 8 epilogue warps
constexpr int kCvGroups = 2;     // epilogue groups of four warps (alternate output rows)

template <int NDIM>
struct CvGeom {
  static constexpr int NZ = NDIM == 3 ? 3 : 1;       // rows per set (z - 1, z, z + 1)
  static constexpr int NS = NDIM == 3 ? 6 : 8;       // sets in the ring
  static constexpr int MINB = NDIM == 3 ? 1 : 2;     // CTAs per SM
  static constexpr int NACC = 8;                      // output rows in TMEM
  static constexpr int T = net_taps(NDIM);
  static constexpr int KB = T * kNetC;                // GEMM K
  static constexpr int NG = T / 3;                    // (dz, ox) groups of B: 96 x 32 each
  static constexpr int SET = NZ * kCvRow;
  static constexpr int OFF_A = (64 * KB + 1023) / 1024 * 1024;
  static constexpr int OFF_BAR = OFF_A + NS * SET;
  // full[NS], empty[NS], accf[NACC], acce[NACC], fin; the TMEM slot and
  // abort word; the 32 biases
  static constexpr int OFF_BIAS = OFF_BAR + (2 * NS + 2 * NACC + 1) * 8 + 16;
  static constexpr int SMEM = OFF_BIAS + 32 * 4;
  static_assert(SMEM <= 227 * 1024, "shared memory");
};

struct CvItem {
  int b, z, x0, ya, nrows;
};

__device__ __forceinline__ CvItem cv_item(int64_t item, const NetShape &sh, int tiles_x, int nchunk,
                                          int chunk) {
  CvItem it;
  const int tx = (int)(item % tiles_x);
  int64_t r = item / tiles_x;
  const int yc = (int)(r % nchunk);
  r /= nchunk;
  it.z = (int)(r % sh.nz);
  it.b = (int)(r / sh.nz);
  it.x0 = tx * 128;
  it.ya = yc * chunk;
  it.nrows = min(chunk, sh.ny - it.ya);
  return it;
}

}  // namespace

// MODE 0: forward epilogue (bias, zout, GELU, replicated store into outpad);
// MODE 1: the data gradient: outpad = raw x gelu'(zin) inside the grid, outraw
// on its faces.
template <int NDIM, int MODE>
__global__ void __launch_bounds__(kCvThreads, CvGeom<NDIM>::MINB)
    net_conv_rows_k(const __grid_constant__ CUtensorMap in_map, const bf16 *__restrict__ Wx,
                    const float *__restrict__ bias, NetShape sh, int chunk, bf16 *__restrict__ zout,
                    bf16 *__restrict__ outpad, float *__restrict__ outraw, const bf16 *__restrict__ zin,
                    int *status) {
  using Gm = CvGeom<NDIM>;
  constexpr int NS = Gm::NS, NZ = Gm::NZ, NG = Gm::NG, KB = Gm::KB;
  constexpr int NACC = Gm::NACC;
  extern __shared__ __align__(1024) unsigned char sm[];
  unsigned char *sB = sm;
  unsigned char *sA = sm + Gm::OFF_A;
  uint64_t *full = reinterpret_cast<uint64_t *>(sm + Gm::OFF_BAR);
  uint64_t *empty = full + NS;
  uint64_t *accf = empty + NS;
  uint64_t *acce = accf + NACC;
  uint64_t *fin = acce + NACC;
  uint32_t *tslot = reinterpret_cast<uint32_t *>(fin + 1);
  volatile int &abort_flag = *reinterpret_cast<volatile int *>(tslot + 1);
  float *sbias = reinterpret_cast<float *>(sm + Gm::OFF_BIAS);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < 32) sbias[tid] = MODE == 0 ? bias[tid] : 0.0f;

  // B operand for the CTA's lifetime: per group (dz, ox) 96 rows n = (2 - dy)
  // * 32 + output channel, dy the tap's row (0..2), by 32 input channels,
  // canonical K-major
  for (int i = tid; i < NG * 96 * 4; i += kCvThreads) {
    const int k8 = i & 3, n = (i >> 2) % 96, gq = (i >> 2) / 96;
    const int t = (gq / 3) * 9 + (2 - n / 32) * 3 + gq % 3;
    *reinterpret_cast<uint4 *>(sB + gq * 96 * 64 + tc_kmajor_off(n, k8 * 8, 4)) =
        *reinterpret_cast<const uint4 *>(Wx + (int64_t)(n % 32) * KB + t * 32 + k8 * 8);
  }
  if (tid == 0) {
    tma_prefetch_desc(&in_map);
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < NACC; ++a) {
      mbar_init(&accf[a], 1);
      mbar_init(&acce[a], 4);
    }
    mbar_init(fin, 1);
    fence_mbar_init();
    abort_flag = 0;
  }
  if (warp == 1) {
    tmem_alloc(tslot, 32 * NACC);
    tmem_relinquish();
  }
  fence_proxy_async_smem();  // B (generic writes) before the MMAs read it
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  const int tiles_x = (sh.nx + 127) / 128;
  const int nchunk = (sh.ny + chunk - 1) / chunk;
  const int64_t items = (int64_t)sh.batch * sh.nz * nchunk * tiles_x;

  if (warp == 0) {
    // ---------------------------------------------------------- TMA loads --
    if (lane == 0) {
      uint32_t i = 0;  // row sets issued
      bool ok = true;
      for (int64_t item = blockIdx.x; item < items && ok; item += gridDim.x) {
        const CvItem it = cv_item(item, sh, tiles_x, nchunk, chunk);
        for (int r = 0; r < it.nrows + 2 && ok; ++r, ++i) {
          const int s = (int)(i % NS);
          if (i >= (uint32_t)NS && !mbar_wait_bounded(&empty[s], ((i / NS) - 1) & 1u)) {
            ok = false;
            break;
          }
          if (abort_flag) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&full[s], NZ * kCvBox);
          for (int dz = 0; dz < NZ; ++dz) {
            // padded row (z + dz, ya + r) from padded column x0 (= cell x0 - 1)
            const int64_t p0 = sh.p(it.b, NDIM == 3 ? it.z + dz : 0, it.ya + r, it.x0);
            tma_load_2d(sA + s * Gm::SET + dz * kCvRow, &in_map, &full[s], 0, (int)p0);
          }
        }
      }
      if (!ok && !abort_flag) {
        report_timeout(status);
        abort_flag = 1;
      }
      // never leave with a copy in flight
      for (uint32_t v = i > (uint32_t)NS ? i - NS : 0; v < i; ++v)
        mbar_wait_bounded(&full[v % NS], (v / NS) & 1u);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------- MMAs --
    if (lane == 0) {
      const uint64_t a_desc0 = tc_smem_desc_sw64(sA, 16, 512);  // A rows: SBO 8 px
      const uint64_t b_desc0 = tc_smem_desc(sB, 128, 512);      // B: canonical K-major, 32 channels
      // (dz, ox) and channel half gk: offsets of A's and B's start addresses
      auto a_off = [](int gk) {
        return (uint32_t)(((gk / 6) * kCvRow + (gk / 2 % 3) * 64 + (gk & 1) * 32) >> 4);
      };
      auto b_off = [](int gk) { return (uint32_t)(((gk >> 1) * 96 * 64 + (gk & 1) * 256) >> 4); };
      constexpr uint32_t idesc0 = tc_idesc_bf16_f32(128, 0);  // + (N / 32) << 19
      uint32_t i = 0, q0 = 0;  // row sets used; output rows of the items before this one
      bool ok = true;
      for (int64_t item = blockIdx.x; item < items && ok; item += gridDim.x) {
        const CvItem it = cv_item(item, sh, tiles_x, nchunk, chunk);
        for (int r = 0; r < it.nrows + 2; ++r, ++i) {
          const int s = (int)(i % NS);
          // the block that this row starts must have been read
          if (r < it.nrows) {
            const uint32_t q = q0 + r;
            if (q >= (uint32_t)NACC && !mbar_wait_bounded(&acce[q % NACC], (q / NACC - 1) & 1u)) ok = false;
          }
          if (ok && !mbar_wait_bounded(&full[s], (i / NS) & 1u)) ok = false;
          if (!ok || abort_flag) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t da = a_desc0 + (uint32_t)(s * (Gm::SET >> 4));
          // output rows j0 .. j1 of the item, row j through tap dy = r - j
          // (block 2 - dy of B's rows); segment 1 is what wraps around the ring
          const int j0 = max(r - 2, 0), j1 = min(r, it.nrows - 1);
          const uint32_t blk = (q0 + j0) % NACC;
          const int c0 = min(j1 - j0 + 1, NACC - (int)blk), c1 = j1 - j0 + 1 - c0;
          const uint32_t d0 = tmem + blk * 32;
          const uint64_t db0 = b_desc0 + (uint32_t)(((2 - (r - j0)) * 4 * 512) >> 4);
          const uint64_t db1 = db0 + (uint32_t)((c0 * 4 * 512) >> 4);
          const uint32_t id0 = idesc0 + ((uint32_t)c0 << 19), id1 = idesc0 + ((uint32_t)c1 << 19);
          // first the MMA that starts row r from zero, and its older rows
          const int fresh = r < it.nrows ? 1 : 0;
          if (c1 == 0) {
            if (fresh)
              tc_mma_bf16(d0 + (c0 - 1) * 32, da, db0 + (uint32_t)(((c0 - 1) * 4 * 512) >> 4),
                          idesc0 + (1u << 19), false);
            if (c0 > fresh) tc_mma_bf16(d0, da, db0, idesc0 + ((uint32_t)(c0 - fresh) << 19), true);
#pragma unroll
            for (int gk = 1; gk < 2 * NG; ++gk)
              tc_mma_bf16(d0, da + a_off(gk), db0 + b_off(gk), id0, true);
          } else {
            tc_mma_bf16(d0, da, db0, id0, true);
            if (fresh)
              tc_mma_bf16(tmem + (c1 - 1) * 32, da, db1 + (uint32_t)(((c1 - 1) * 4 * 512) >> 4),
                          idesc0 + (1u << 19), false);
            if (c1 > fresh) tc_mma_bf16(tmem, da, db1, idesc0 + ((uint32_t)(c1 - fresh) << 19), true);
#pragma unroll
            for (int gk = 1; gk < 2 * NG; ++gk) {
              tc_mma_bf16(d0, da + a_off(gk), db0 + b_off(gk), id0, true);
              tc_mma_bf16(tmem, da + a_off(gk), db1 + b_off(gk), id1, true);
            }
          }
          tc_commit(&empty[s]);
          if (r >= 2) tc_commit(&accf[(q0 + r - 2) % NACC]);
        }
        q0 += it.nrows;
      }
      if (!ok && !abort_flag) {
        report_timeout(status);
        abort_flag = 1;
      }
      // every MMA issued has completed before the accumulator is freed
      tc_commit(fin);
      mbar_wait_bounded(fin, 0);
    }
  } else {
    // -------------------------------------------------------- epilogue --
    const int q = warp & 3;  // TMEM lane quarter of this warp
    const uint32_t grp = (uint32_t)(warp - 2) >> 2;
    uint32_t q0 = 0;  // output rows of the items before this one
    bool ok = true;
    for (int64_t item = blockIdx.x; item < items && ok; item += gridDim.x) {
      const CvItem it = cv_item(item, sh, tiles_x, nchunk, chunk);
      for (int j = (int)((grp + q0) & 1u); j < it.nrows; j += kCvGroups) {
        const uint32_t buf = (q0 + j) % NACC;
        const uint32_t par = ((q0 + j) / NACC) & 1u;
        const int x = it.x0 + q * 32 + lane;
        const int y = it.ya + j;
        bool inner = false;
        uint4 zw[4];
        if (MODE == 1) {  // the pre-activations, ahead of the wait
          inner = x > 0 && x < sh.nx - 1 && y > 0 && y < sh.ny - 1 &&
                  (NDIM == 2 || (it.z > 0 && it.z < sh.nz - 1));
          if (inner) {
            const bf16 *zs = zin + sh.u(it.b, it.z, y, x) * kNetC;
            ld_global32(zs, zw[0], zw[1]);
            ld_global32(zs + 16, zw[2], zw[3]);
          }
        }
        const bool got = mbar_wait_bounded(&accf[buf], par);
        if (__any_sync(0xffffffffu, !got || abort_flag)) {  // the warp leaves together
          ok = false;
          break;
        }
        tc_fence_after();
        float v[32];
        tmem_ld32(tmem + buf * 32 + ((uint32_t)(q * 32) << 16), v);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce[buf]);
        if (x < sh.nx) {
          const int64_t pu = sh.u(it.b, it.z, y, x);
          if (MODE == 0) {
            uint64_t xv[16];
#pragma unroll
            for (int c = 0; c < 16; ++c)
              xv[c] = add2(pack2(v[2 * c], v[2 * c + 1]), reinterpret_cast<const uint64_t *>(sbias)[c]);
            if (zout) {
#pragma unroll
              for (int c = 0; c < 16; ++c) unpack2(xv[c], v[2 * c], v[2 * c + 1]);
              bf16 *dz = zout + pu * kNetC;
              st_global32(dz, pack8_bf16(v), pack8_bf16(v + 8));
              st_global32(dz + 16, pack8_bf16(v + 16), pack8_bf16(v + 24));
            }
#pragma unroll
            for (int c = 0; c < 16; ++c) unpack2(net_gelu_fast2(xv[c]), v[2 * c], v[2 * c + 1]);
            store_replicated<NDIM>(outpad, sh, it.b, it.z, y, x, v);
          } else if (inner) {
            bf16 *d = outpad + sh.ps(it.b, it.z, y, x, 0, 0, 0) * kNetC;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              float zv[8];
              unpack8_bf16(zw[c], zv);
#pragma unroll
              for (int e = 0; e < 8; e += 2)
                unpack2(mul2(pack2(v[8 * c + e], v[8 * c + e + 1]), net_gelu_grad2(pack2(zv[e], zv[e + 1]))),
                        zv[e], zv[e + 1]);
              zw[c] = pack8_bf16(zv);
            }
            st_global32(d, zw[0], zw[1]);
            st_global32(d + 16, zw[2], zw[3]);
          } else {
            float4 *d = reinterpret_cast<float4 *>(outraw + pu * kNetC);
#pragma unroll
            for (int c = 0; c < 8; ++c)
              d[c] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
          }
        }
      }
      q0 += it.nrows;
    }
    if (!ok && lane == 0 && !abort_flag) {
      report_timeout(status);
      abort_flag = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 32 * NACC);
}

// ------------------------------------------------------------------ host ---
template <int NDIM, int MODE>
static cudaError_t conv_rows_t(const bf16 *in, const bf16 *Wx, const float *bias,
                               const NetShape &sh, bf16 *zout, bf16 *outpad, float *outraw,
                               const bf16 *zin, int *status, int num_sms, cudaStream_t s) {
  using Gm = CvGeom<NDIM>;
  static KernelSetup ks;
  int occ = 1;
  cudaError_t e0 = kernel_setup(ks, (const void *)net_conv_rows_k<NDIM, MODE>, kCvThreads, Gm::SMEM,
                                &occ, 100);
  if (e0 != cudaSuccess) return e0;
  // the register budget of __launch_bounds__ guarantees MINB CTAs per SM
  // (the shared memory fits as well); the query may report fewer
  occ = std::max(occ, Gm::MINB);
  // the padded activations as a 2D tensor {32 channels, padded pixels}
  const int64_t P = sh.padded_cells();
  if (P + 2 * kCvPix >= (int64_t)INT32_MAX) return cudaErrorInvalidValue;
  EncodeTiledFn fn = ac_encode_fn();
  if (!fn) return cudaErrorNotSupported;
  CUtensorMap map;
  const cuuint64_t dims[2] = {(cuuint64_t)kNetC, (cuuint64_t)P};
  const cuuint64_t strides[1] = {(cuuint64_t)kNetC * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kNetC, (cuuint32_t)kCvPix}, es[2] = {1, 1};
  if (fn(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16 *>(in), dims, strides, box, es,
         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  // rows per item: about two items per resident CTA, at least 4 rows (each
  // item loads its rows + 2)
  const int64_t slots = (int64_t)std::max(1, num_sms) * occ;
  const int64_t columns = (int64_t)sh.batch * sh.nz * ((sh.nx + 127) / 128);
  int chunk = (int)std::min<int64_t>(sh.ny, std::max<int64_t>(4, (columns * sh.ny + 2 * slots - 1) / (2 * slots)));
  const int nchunk = (sh.ny + chunk - 1) / chunk;
  const int64_t items = columns * nchunk;
  const int grid = (int)std::min<int64_t>(items, slots);
  net_conv_rows_k<NDIM, MODE><<<grid, kCvThreads, Gm::SMEM, s>>>(map, Wx, bias, sh, chunk, zout,
                                                                  outpad, outraw, zin, status);
  return cudaGetLastError();
}

cudaError_t net_conv_rows(int mode, const bf16 *in, const bf16 *Wx, const float *bias,
                          const NetShape &sh, bf16 *zout, bf16 *outpad, float *outraw, const bf16 *zin,
                          int *status, int num_sms, cudaStream_t s) {
  if (sh.ndim == 3)
    return mode == 0 ? conv_rows_t<3, 0>(in, Wx, bias, sh, zout, outpad, outraw, zin, status, num_sms, s)
                     : conv_rows_t<3, 1>(in, Wx, bias, sh, zout, outpad, outraw, zin, status, num_sms, s);
  return mode == 0 ? conv_rows_t<2, 0>(in, Wx, bias, sh, zout, outpad, outraw, zin, status, num_sms, s)
                   : conv_rows_t<2, 1>(in, Wx, bias, sh, zout, outpad, outraw, zin, status, num_sms, s);
}

}  // namespace ac
