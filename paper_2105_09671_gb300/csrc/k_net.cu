// Kernels of the learned 16-step jump network (layout and definition in
// net.cuh).  Activations are BF16 with FP32 accumulation.
//
// Storage: every activation a_l that feeds a convolution is kept *padded*:
// [batch][nz+2][ny+2][nx+2][32] (2D: [batch][1][ny+2][nx+2][32]) with the
// ghost ring holding the replicated boundary cell (the zero-Neumann ghost),
// written by the layer that produces a_l.  Gradients wrt pre-activations are
// kept padded with a zero ghost ring.  So every tap of every convolution
// reads an in-bounds, unclamped shifted row.
//
//   net_first_fwd     1 -> 32 channels, CUDA cores (K = 9 / 27 is too short)
//   net_conv_rows     out[p][n] = sum_t sum_c in[p+t][c] Wx[n][t][c] on the
//                     tensor cores (k_net_conv.cu: TMA row ring, tcgen05,
//                     accumulators in TMEM); forward (bias, GELU, ghost
//                     writes) and the data gradient (flipped taps,
//                     transposed weights, x gelu')
//   net_dgrad_faces   the data gradient of face cells: adds the gradient of
//                     the ghost cells that copy them (adjoint of replicate
//                     padding), x gelu'
//   net_wgrad         dW[t][ci][co] = sum_p a[p+t][ci] g[p][co] on the
//                     tensor cores, reduced over pixels, and the bias
//                     gradient (k_net_wgrad.cu)
//   net_last_fwd/bwd, net_first_wgrad   the 1-channel ends, CUDA cores
//   net_adam, net_pack                  optimiser and BF16 weight layouts
#include <cuda_bf16.h>

#include <algorithm>

#include "kernels.h"
#include "net.cuh"

namespace ac {

// ------------------------------------------------------------ first layer --
// A thread per cell of a 32 x 8 tile of one z, packed FP32 pairs of channels;
// a block takes one tile after another.  Bound by latency (the taps' loads, then
// 16 chains of multiply-adds): three blocks to an SM in 80 registers, two where
// that would spill.  1024^2 31 us (36 with 84 registers and two blocks), 32 x
// 256^2 with the pre-activations 66 (81).  Weights in registers, a quarter of
// the channels a lane, and cells marching along y: 41 and 87 us.
template <int NDIM, bool TRAIN>
constexpr int first_blocks() { return NDIM == 3 && TRAIN ? 2 : 3; }

template <int NDIM, bool TRAIN>
__global__ void __launch_bounds__(256, first_blocks<NDIM, TRAIN>())
    net_first_fwd_k(const float *__restrict__ phi, const float *__restrict__ params, int64_t w_off,
                    int64_t b_off, NetShape sh, bf16 *__restrict__ z1, bf16 *__restrict__ a1pad) {
  constexpr int T = net_taps(NDIM);
  __shared__ __align__(16) float w[T * kNetC];
  __shared__ __align__(16) float bb[kNetC];
  for (int i = threadIdx.x; i < T * kNetC; i += blockDim.x) w[i] = params[w_off + i];
  if (threadIdx.x < kNetC) bb[threadIdx.x] = params[b_off + threadIdx.x];
  __syncthreads();
  const uint32_t tiles_x = (uint32_t)(sh.nx + 31) / 32, tiles_y = (uint32_t)(sh.ny + 7) / 8;
  const uint32_t tiles = tiles_x * tiles_y * (uint32_t)sh.batch * (uint32_t)sh.nz;
  for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const uint32_t r = tile / tiles_x, bz = r / tiles_y;
    const int x = (int)(tile - r * tiles_x) * 32 + (threadIdx.x & 31);
    const int y = (int)(r - bz * tiles_y) * 8 + (threadIdx.x >> 5);
    if (x >= sh.nx || y >= sh.ny) continue;
    const int b = NDIM == 2 ? (int)bz : (int)(bz / (uint32_t)sh.nz), z = NDIM == 2 ? 0 : (int)(bz - (uint32_t)b * sh.nz);
    uint64_t acc[kNetC / 2];
#pragma unroll
    for (int c = 0; c < kNetC / 2; ++c) acc[c] = reinterpret_cast<const uint64_t *>(bb)[c];
#pragma unroll
    for (int t = 0; t < T; ++t) {
      const int ox = t % 3 - 1, oy = (t / 3) % 3 - 1, oz = NDIM == 3 ? t / 9 - 1 : 0;
      const int xx = min(max(x + ox, 0), sh.nx - 1), yy = min(max(y + oy, 0), sh.ny - 1);
      const int zz = NDIM == 3 ? min(max(z + oz, 0), sh.nz - 1) : 0;
      const float v = phi[sh.u(b, zz, yy, xx)];
      const uint64_t vv = pack2(v, v);
#pragma unroll
      for (int c = 0; c < kNetC / 2; c += 2) {  // 16-byte weight reads (broadcast)
        const ulonglong2 wv = *reinterpret_cast<const ulonglong2 *>(w + t * kNetC + 2 * c);
        acc[c] = fma2(vv, wv.x, acc[c]);
        acc[c + 1] = fma2(vv, wv.y, acc[c + 1]);
      }
    }
    float a[kNetC];
    if (TRAIN) {
#pragma unroll
      for (int c = 0; c < kNetC / 2; ++c) unpack2(acc[c], a[2 * c], a[2 * c + 1]);
      bf16 *dz = z1 + sh.u(b, z, y, x) * kNetC;
      st_global32(dz, pack8_bf16(a), pack8_bf16(a + 8));
      st_global32(dz + 16, pack8_bf16(a + 16), pack8_bf16(a + 24));
    }
#pragma unroll
    for (int c = 0; c < kNetC / 2; ++c) unpack2(net_gelu_fast2(acc[c]), a[2 * c], a[2 * c + 1]);
    store_replicated<NDIM>(a1pad, sh, b, z, y, x, a);
  }
}

// ------------------------------------------------------------- last layer --
// z6 = conv(a5, W6) + b6 (32 -> 1 channel) and phi_hat = phi + s z6; in
// training also the scaled residual's gradient g6 and the loss sum.  A block
// covers 32 x 32 cells of one z, a thread 4 cells above one another: the
// padded pixels of one plane at a time are staged in shared memory with
// asynchronous 16-byte copies, all in flight at once (pixel stride 80 bytes:
// conflict-free 16-byte reads by consecutive lanes), and a pixel read serves the up to 3 cells of the
// thread that it is a tap of, a weight read all 4 (one cell a thread read each
// pixel 9 times and all weights: 64 us at 1024^2).
constexpr int kLastTX = 32, kLastRows = 4, kLastTY = 8 * kLastRows, kLastPix = 5;  // uint4 per staged pixel (4 + pad)

template <int NDIM>
__host__ __device__ constexpr int last_smem_bytes() {
  return (kLastTY + 2) * (kLastTX + 2) * kLastPix * 16 + net_taps(NDIM) * kNetC * 4;
}

// Two BF16 values as a packed FP32 pair.
__device__ __forceinline__ uint64_t bf16_pair(uint32_t w) {
  return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

template <int NDIM, bool TRAIN>
__global__ void __launch_bounds__(256) net_last_fwd_k(const bf16 *__restrict__ a5pad,
                                                      const float *__restrict__ params, int64_t w_off,
                                                      int64_t b_off, NetShape sh,
                                                      const float *__restrict__ phi, float scale,
                                                      float *__restrict__ phihat,
                                                      const float *__restrict__ target,
                                                      float *__restrict__ g6, double *loss_acc) {
  constexpr int T = net_taps(NDIM);
  constexpr int NZR = NDIM == 3 ? 3 : 1;
  constexpr int RW = kLastTX + 2, RH = kLastTY + 2;
  extern __shared__ __align__(16) unsigned char lsm[];
  uint4 *tile = reinterpret_cast<uint4 *>(lsm);                          // [RH][RW][kLastPix]
  float *w = reinterpret_cast<float *>(lsm + RH * RW * kLastPix * 16);   // [T][32]
  __shared__ double red[8];
  for (int i = threadIdx.x; i < T * kNetC; i += blockDim.x) w[i] = params[w_off + i];
  const float b6 = params[b_off];
  const float inv_n = 1.0f / (float)sh.cells();
  const int tiles_x = (sh.nx + kLastTX - 1) / kLastTX, tiles_y = (sh.ny + kLastTY - 1) / kLastTY;
  const int64_t items = (int64_t)sh.batch * sh.nz * tiles_y * tiles_x;
  const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
  double lsum = 0.0;
  for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const int tx = (int)(item % tiles_x);
    int64_t r = item / tiles_x;
    const int ty = (int)(r % tiles_y);
    r /= tiles_y;
    const int z = (int)(r % sh.nz), b = (int)(r / sh.nz);
    const int x0 = tx * kLastTX, y0 = ty * kLastTY;
    uint64_t acc[kLastRows];
#pragma unroll
    for (int q = 0; q < kLastRows; ++q) acc[q] = 0;
    for (int dz = 0; dz < NZR; ++dz) {
      __syncthreads();  // the previous plane (and w) is complete / released
      // padded pixels (xp, yp) = (x0 + i, y0 + j), i < RW, j < RH, of plane z + dz
      for (int i = threadIdx.x; i < RH * RW * 4; i += blockDim.x) {
        const int c = i & 3, q = i >> 2;
        const int px = q % RW, row = q / RW;
        const int xp = x0 + px, yp = y0 + row;
        const bool in = xp < sh.px() && yp < sh.py();
        cp_async16(tile + q * kLastPix + c,
                   a5pad + (in ? sh.p(b, NDIM == 3 ? z + dz : 0, yp, xp) * kNetC + c * 8 : 0), in);
      }
      cp_async_wait();
      __syncthreads();
#pragma unroll
      for (int ox = 0; ox < 3; ++ox)
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          uint64_t wv[3][4];  // 8 channels of the three oy
#pragma unroll
          for (int oy = 0; oy < 3; ++oy) {
            const float *wp = w + (dz * 9 + oy * 3 + ox) * kNetC + c * 8;
            const ulonglong2 lo = *reinterpret_cast<const ulonglong2 *>(wp);
            const ulonglong2 hi = *reinterpret_cast<const ulonglong2 *>(wp + 4);
            wv[oy][0] = lo.x; wv[oy][1] = lo.y; wv[oy][2] = hi.x; wv[oy][3] = hi.y;
          }
#pragma unroll
          for (int j = 0; j < kLastRows + 2; ++j) {
            const uint4 u = tile[((wy * kLastRows + j) * RW + lane + ox) * kLastPix + c];
            const uint64_t a[4] = {bf16_pair(u.x), bf16_pair(u.y), bf16_pair(u.z), bf16_pair(u.w)};
#pragma unroll
            for (int oy = 0; oy < 3; ++oy) {
              const int q = j - oy;  // the cell whose tap oy this row is
              if (q < 0 || q >= kLastRows) continue;
#pragma unroll
              for (int e = 0; e < 4; ++e) acc[q] = fma2(a[e], wv[oy][e], acc[q]);
            }
          }
        }
    }
    const int x = x0 + lane;
#pragma unroll
    for (int q = 0; q < kLastRows; ++q) {
      const int y = y0 + wy * kLastRows + q;
      if (x >= sh.nx || y >= sh.ny) continue;
      float even, odd;
      unpack2(acc[q], even, odd);
      const int64_t i = sh.u(b, z, y, x);
      const float ph = phi[i] + scale * (b6 + (even + odd));
      phihat[i] = ph;
      if (TRAIN) {
        const float rr = (ph - target[i]) / scale;
        g6[i] = 2.0f * rr * inv_n;
        lsum += (double)rr * (double)rr;
      }
    }
  }
  if (TRAIN) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if (lane == 0) red[wy] = lsum;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s2 = 0.0;
      for (int w2 = 0; w2 < (int)(blockDim.x >> 5); ++w2) s2 += red[w2];
      atomicAdd(loss_acc, s2);
    }
  }
}

// Warp per face cell: g_{l-1} = (raw + ghost-cell gradients folded in) x
// gelu'(z_{l-1}).  raw[p] = sum_t W[t]^T g[p - t] comes from the tensor-core
// pass; a face cell also receives the gradient of each ghost cell that
// replicates it: lane ci sums W[t][ci][co] g[p - t][co] over the taps that
// read a cell of the grid.  Bound by latency: a warp meets 7 cells one after
// the other at 32 x 256^2 pixels (30 us).  So the gradients of a plane's nine
// taps are loaded together and shared through shared memory (one load at a
// time, and a shuffle per value: 50 us), and the cells are enumerated in 32
// bits (64-bit divisions: 41 us).
constexpr int kFacesThreads = 512;
template <int NDIM>
__host__ __device__ constexpr int faces_smem() {
  return net_taps(NDIM) * kNetC * kNetC * 4 + kFacesThreads / 32 * 9 * kNetC * 4;
}

template <int NDIM>
__global__ void __launch_bounds__(kFacesThreads) net_dgrad_faces_k(const float *__restrict__ raw,
                                                                   const bf16 *__restrict__ gpad,
                                                                   const float *__restrict__ params,
                                                                   int64_t w_off, NetShape sh,
                                                                   const bf16 *__restrict__ zprev,
                                                                   bf16 *__restrict__ gprevpad) {
  constexpr int T = net_taps(NDIM);
  // W[t][ci][co], the four-float groups of a row at (group ^ ci % 8) so that
  // eight lanes read eight different ones; then 9 x 32 gradients per warp
  extern __shared__ __align__(16) float wsm[];
  for (int i = threadIdx.x; i < T * kNetC * kNetC / 4; i += blockDim.x) {
    const int ci = i / 8 % kNetC;
    reinterpret_cast<float4 *>(wsm)[(i & ~7) + ((i ^ ci) & 7)] = reinterpret_cast<const float4 *>(params + w_off)[i];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  float *gs = wsm + T * kNetC * kNetC + (threadIdx.x >> 5) * 9 * kNetC;
  const int warps = (int)(gridDim.x * (blockDim.x >> 5));
  // face cells of an image: the rows on y and z faces whole, then the two end
  // cells of the other rows (in 32 bits: the layers' padded cells are fewer
  // than 2^31)
  const int fy = min(sh.ny, 2), fz = NDIM == 3 ? min(sh.nz, 2) : 0, fx = min(sh.nx, 2);
  const int whole = (fz * sh.ny + (sh.nz - fz) * fy) * sh.nx;
  const int per = whole + (sh.nz - fz) * (sh.ny - fy) * fx;
  for (int64_t u = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); u < (int64_t)per * sh.batch; u += warps) {
    const int b = (int)((uint32_t)u / (uint32_t)per);
    int f = (int)((uint32_t)u % (uint32_t)per);
    int z, y, x;
    if (f < whole) {
      x = f % sh.nx;
      f /= sh.nx;
      if (f < fz * sh.ny) {
        z = f < sh.ny ? 0 : sh.nz - 1;
        y = f % sh.ny;
      } else {
        f -= fz * sh.ny;
        z = (NDIM == 3 ? 1 : 0) + f / fy;
        y = f % fy ? sh.ny - 1 : 0;
      }
    } else {
      f -= whole;
      x = f % fx ? sh.nx - 1 : 0;
      f /= fx;
      z = (NDIM == 3 ? 1 : 0) + f / (sh.ny - fy);
      y = 1 + f % (sh.ny - fy);
    }
    const int64_t i = sh.u(b, z, y, x);
    float g = raw[i * kNetC + lane];
    // ghost cells q (outside the grid by one) with clamp(q) == p
    const int gx0 = x == 0 ? -1 : 0, gx1 = x == sh.nx - 1 ? 1 : 0;
    const int gy0 = y == 0 ? -1 : 0, gy1 = y == sh.ny - 1 ? 1 : 0;
    const int gz0 = NDIM == 3 && z == 0 ? -1 : 0, gz1 = NDIM == 3 && z == sh.nz - 1 ? 1 : 0;
    for (int gz = gz0; gz <= gz1; ++gz)
      for (int gy = gy0; gy <= gy1; ++gy)
        for (int gx = gx0; gx <= gx1; ++gx) {
          if (gx == 0 && gy == 0 && gz == 0) continue;
          const int qx = x + gx, qy = y + gy, qz = z + gz;
          // gradient of the ghost cell q: sum_t W[t][ci = lane][co] g[q - t][co]
          uint64_t acc = 0;
          for (int tz = 0; tz < T; tz += 9) {
            const int sz = NDIM == 3 ? qz + 1 - tz / 9 : 0;
            if (NDIM == 3 && (sz < 0 || sz >= sh.nz)) continue;
            bf16 gv[9] = {};
            const bf16 *gq = gpad + sh.ps(b, sz, qy, qx, 0, 0, 0) * kNetC + lane;
#pragma unroll
            for (int t = 0; t < 9; ++t) {
              const int sx = qx + 1 - t % 3, sy = qy + 1 - t / 3;
              if (sx >= 0 && sx < sh.nx && sy >= 0 && sy < sh.ny)
                gv[t] = gq[((int64_t)(1 - t / 3) * sh.px() + (1 - t % 3)) * kNetC];
            }
            __syncwarp();
#pragma unroll
            for (int t = 0; t < 9; ++t) gs[t * kNetC + lane] = __bfloat162float(gv[t]);
            __syncwarp();
#pragma unroll
            for (int t = 0; t < 9; ++t) {
              const int sx = qx + 1 - t % 3, sy = qy + 1 - t / 3;
              if (sx < 0 || sx >= sh.nx || sy < 0 || sy >= sh.ny) continue;
              const ulonglong2 *wr = reinterpret_cast<const ulonglong2 *>(wsm + ((tz + t) * kNetC + lane) * kNetC);
              const ulonglong2 *gr = reinterpret_cast<const ulonglong2 *>(gs + t * kNetC);
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                const ulonglong2 w = wr[k ^ (lane & 7)], v = gr[k];
                acc = fma2(w.x, v.x, acc);
                acc = fma2(w.y, v.y, acc);
              }
            }
          }
          float even, odd;
          unpack2(acc, even, odd);
          g += even + odd;
        }
    const float zv = __bfloat162float(zprev[i * kNetC + lane]);
    gprevpad[sh.ps(b, z, y, x, 0, 0, 0) * kNetC + lane] = __float2bfloat16_rn(g * net_gelu_grad(zv));
  }
}

// ---------------------------------------------- backward of the end layers --
// A block covers tiles of 32 x 8 cells of one z.  A channel-per-lane pass over
// staged shared memory forms the weight gradients: a half warp (2 channels a
// lane) takes 16 cells of a row, and its window of taps is read from shared
// memory.  kEndRow pads the pixel rows so that a warp's two half warps, on
// adjacent rows, use different banks.
constexpr int kEndTX = 32, kEndTY = 8;
constexpr int kEndRow = kEndTX + 3;   // pixels per staged row of activations (34 used; 64 bytes each)
constexpr int kEndRow1 = kEndTX + 4;  // floats per staged row of a field (34 used; whole 16-byte groups)

template <int NDIM>
__host__ __device__ constexpr int end_planes() { return NDIM == 3 ? 3 : 1; }

// Adds dw[t] (this lane's two channels) of all half warps of the block in
// shared memory and then to the global gradient, float by float.
template <int T>
__device__ __forceinline__ void end_reduce(float *acc, const uint64_t *dw, float *gw) {
  const int cl = (threadIdx.x & 15) * 2;
  for (int i = threadIdx.x; i < T * kNetC; i += blockDim.x) acc[i] = 0.f;
  __syncthreads();
#pragma unroll
  for (int t = 0; t < T; ++t) {
    float a, b;
    unpack2(dw[t], a, b);
    atomicAdd(acc + t * kNetC + cl, a);
    atomicAdd(acc + t * kNetC + cl + 1, b);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < T * kNetC; i += blockDim.x) atomicAdd(gw + i, acc[i]);
}

__device__ __forceinline__ float2 ld_bf2(const unsigned char *p) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p));
}

template <int NDIM>
__host__ __device__ constexpr int last_bwd_smem() {
  return end_planes<NDIM>() * (kEndTY + 2) * kEndRow * 64 + end_planes<NDIM>() * (kEndTY + 2) * kEndRow1 * 4 +
         net_taps(NDIM) * kNetC * 4;
}

// Gradient of the last layer's weights and bias, and the gradient wrt z5:
// g5 = (sum_t W6[t] S_t) x gelu'(z5), S_t(p) the sum of g6 over the cells
// whose tap t reads p (with replicate padding a boundary cell is also read
// in the place of the ghosts that copy it).
// First pass, one thread per cell: S_t from the staged g6 (zero outside the
// grid): the cell at p - t, and per axis, where p is a face cell, the cell
// at offset 0 once more for the tap that points out of the grid.
// Second pass: dW6[t][c] += a5[p + t][c] g6[p] from the staged a5.
// Bound by instruction issue and latency (about 9 + 9 multiply-adds and a
// gelu' per cell and channel, on two channels an instruction; 16 warps to an SM
// in 128 registers).  32 x 256^2 cells: 160 us; with scalar arithmetic 196, the
// copies not asynchronous 245, one warp per cell and every operand read from
// global memory 2818.
template <int NDIM>
__global__ void __launch_bounds__(256, 2) net_last_bwd_k(const float *__restrict__ g6,
                                                         const float *__restrict__ params, int64_t w_off,
                                                         NetShape sh, const bf16 *__restrict__ z5,
                                                         const bf16 *__restrict__ a5pad,
                                                         bf16 *__restrict__ gz5pad,
                                                         float *__restrict__ grads, int64_t gw_off,
                                                         int64_t gb_off) {
  constexpr int T = net_taps(NDIM), NZR = end_planes<NDIM>(), RW = kEndTX + 2, RH = kEndTY + 2;
  extern __shared__ __align__(16) unsigned char lsm[];
  unsigned char *ta = lsm;                                                   // [NZR][RH][kEndRow] pixels
  float *tg = reinterpret_cast<float *>(lsm + NZR * RH * kEndRow * 64);       // [NZR][RH][kEndRow1]
  float *w = tg + NZR * RH * kEndRow1;                                        // [T][32]
  for (int i = threadIdx.x; i < T * kNetC; i += blockDim.x) w[i] = params[w_off + i];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tiles_x = (sh.nx + kEndTX - 1) / kEndTX, tiles_y = (sh.ny + kEndTY - 1) / kEndTY;
  const int64_t items = (int64_t)sh.batch * sh.nz * tiles_y * tiles_x;
  uint64_t dw[T];  // two channels, packed
#pragma unroll
  for (int t = 0; t < T; ++t) dw[t] = 0;
  float db = 0.f;
  for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const int tx = (int)(item % tiles_x);
    int64_t r = item / tiles_x;
    const int ty = (int)(r % tiles_y);
    r /= tiles_y;
    const int z = (int)(r % sh.nz), b = (int)(r / sh.nz);
    const int x0 = tx * kEndTX, y0 = ty * kEndTY;
    __syncthreads();  // the previous item's tiles are released (and w is complete)
    for (int i = threadIdx.x; i < NZR * RH * RW * 4; i += blockDim.x) {
      const int c = i & 3, q = i >> 2;
      const int px = q % RW, row = (q / RW) % RH, dz = q / (RW * RH);
      const bool in = x0 + px < sh.px() && y0 + row < sh.py();
      cp_async16(ta + ((dz * RH + row) * kEndRow + px) * 64 + c * 16,
                 a5pad + (in ? sh.p(b, NDIM == 3 ? z + dz : 0, y0 + row, x0 + px) * kNetC + c * 8 : 0), in);
    }
    for (int i = threadIdx.x; i < NZR * RH * RW; i += blockDim.x) {
      const int px = i % RW, row = (i / RW) % RH, dz = i / (RW * RH);
      const int xx = x0 + px - 1, yy = y0 + row - 1, zz = NDIM == 3 ? z + dz - 1 : 0;
      const bool in = xx >= 0 && xx < sh.nx && yy >= 0 && yy < sh.ny && zz >= 0 && zz < sh.nz;
      cp_async4(tg + (dz * RH + row) * kEndRow1 + px, g6 + (in ? sh.u(b, zz, yy, xx) : 0), in);
    }
    cp_async_wait();
    __syncthreads();
    {
      const int x = x0 + lane, y = y0 + warp;
      if (x < sh.nx && y < sh.ny) {
        // S[t] = g6[p - t], then the faces' second reads axis by axis
        float S[T];
#pragma unroll
        for (int t = 0; t < T; ++t) {
          const int ox = t % 3 - 1, oy = (t / 3) % 3 - 1, oz = NDIM == 3 ? t / 9 - 1 : 0;
          S[t] = tg[((NDIM == 3 ? 1 - oz : 0) * RH + warp + 1 - oy) * kEndRow1 + lane + 1 - ox];
        }
        db += S[T / 2];
        if (NDIM == 3) {
#pragma unroll
          for (int i = 0; i < 9; ++i) {
            const float m = S[(9 + i) % T];
            if (z == 0) S[i] += m;
            if (z == sh.nz - 1) S[(18 + i) % T] += m;
          }
        }
#pragma unroll
        for (int i = 0; i < T / 3; ++i) {  // (plane, ox)
          const int o = (i / 3) * 9 + i % 3;
          const float m = S[o + 3];
          if (y == 0) S[o] += m;
          if (y == sh.ny - 1) S[o + 6] += m;
        }
#pragma unroll
        for (int i = 0; i < T / 3; ++i) {  // (plane, oy)
          const float m = S[3 * i + 1];
          if (x == 0) S[3 * i] += m;
          if (x == sh.nx - 1) S[3 * i + 2] += m;
        }
        const uint4 *zs = reinterpret_cast<const uint4 *>(z5 + sh.u(b, z, y, x) * kNetC);
        uint4 *dst = reinterpret_cast<uint4 *>(gz5pad + sh.ps(b, z, y, x, 0, 0, 0) * kNetC);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint4 zw = zs[c];
          uint64_t g2[4] = {};
#pragma unroll
          for (int t = 0; t < T; ++t) {
            const ulonglong2 wa = *reinterpret_cast<const ulonglong2 *>(w + t * kNetC + c * 8);
            const ulonglong2 wb = *reinterpret_cast<const ulonglong2 *>(w + t * kNetC + c * 8 + 4);
            const uint64_t st = pack2(S[t], S[t]);
            g2[0] = fma2(wa.x, st, g2[0]);
            g2[1] = fma2(wa.y, st, g2[1]);
            g2[2] = fma2(wb.x, st, g2[2]);
            g2[3] = fma2(wb.y, st, g2[3]);
          }
          float zv[8], ga[8];
          unpack8_bf16(zw, zv);
#pragma unroll
          for (int e = 0; e < 4; ++e)
            unpack2(mul2(g2[e], net_gelu_grad2(pack2(zv[2 * e], zv[2 * e + 1]))), ga[2 * e], ga[2 * e + 1]);
          dst[c] = pack8_bf16(ga);
        }
      }
    }
    // second pass: rows 2 (warp % 4) + half, 16 cells from 16 (warp / 4)
    const int row = 2 * (warp & 3) + (lane >> 4), xs = 16 * (warp >> 2);
    const unsigned char *pa = ta + (row * kEndRow + xs) * 64 + (lane & 15) * 4;
    const float *pg = tg + ((NZR / 2) * RH + row + 1) * kEndRow1 + xs + 1;
#pragma unroll(NDIM == 3 ? 2 : 16)
    for (int i = 0; i < 16; ++i) {
      const uint64_t gp = pack2(pg[i], pg[i]);  // (zero outside the grid)
#pragma unroll
      for (int t = 0; t < T; ++t) {
        const int ox = t % 3, oy = (t / 3) % 3, dz = t / 9;
        const float2 a = ld_bf2(pa + ((dz * RH + oy) * kEndRow + i + ox) * 64);
        dw[t] = fma2(pack2(a.x, a.y), gp, dw[t]);
      }
    }
  }
  __syncthreads();
  end_reduce<T>(w, dw, grads + gw_off);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) db += __shfl_xor_sync(0xffffffffu, db, o);
  if (lane == 0) atomicAdd(grads + gb_off, db);
}

template <int NDIM>
__host__ __device__ constexpr int first_wgrad_smem() {
  return kEndTY * kEndRow * 64 + end_planes<NDIM>() * (kEndTY + 2) * kEndRow1 * 4 + net_taps(NDIM) * kNetC * 4;
}

// First-layer weight and bias gradients, dW1[t][c] += phi[p + t] g1[p][c]: g1
// and phi (boundary cells replicated) staged per tile, half warps as above.
template <int NDIM>
__global__ void __launch_bounds__(256, 2) net_first_wgrad_k(const float *__restrict__ phi,
                                                            const bf16 *__restrict__ g1pad, NetShape sh,
                                                            float *__restrict__ grads, int64_t gw_off,
                                                            int64_t gb_off) {
  constexpr int T = net_taps(NDIM), NZR = end_planes<NDIM>(), RW = kEndTX + 2, RH = kEndTY + 2;
  extern __shared__ __align__(16) unsigned char lsm[];
  unsigned char *tg = lsm;                                                 // [kEndTY][kEndRow] pixels
  float *tp = reinterpret_cast<float *>(lsm + kEndTY * kEndRow * 64);       // [NZR][RH][kEndRow1]
  float *acc = tp + NZR * RH * kEndRow1;                                    // [T][32]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tiles_x = (sh.nx + kEndTX - 1) / kEndTX, tiles_y = (sh.ny + kEndTY - 1) / kEndTY;
  const int64_t items = (int64_t)sh.batch * sh.nz * tiles_y * tiles_x;
  uint64_t dw[T], db = 0;  // two channels, packed
#pragma unroll
  for (int t = 0; t < T; ++t) dw[t] = 0;
  for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const int tx = (int)(item % tiles_x);
    int64_t r = item / tiles_x;
    const int ty = (int)(r % tiles_y);
    r /= tiles_y;
    const int z = (int)(r % sh.nz), b = (int)(r / sh.nz);
    const int x0 = tx * kEndTX, y0 = ty * kEndTY;
    __syncthreads();
    for (int i = threadIdx.x; i < kEndTY * kEndTX * 4; i += blockDim.x) {
      const int c = i & 3, px = (i >> 2) % kEndTX, row = (i >> 2) / kEndTX;
      const bool in = x0 + px < sh.nx && y0 + row < sh.ny;
      cp_async16(tg + (row * kEndRow + px) * 64 + c * 16,
                 g1pad + (in ? sh.ps(b, z, y0 + row, x0 + px, 0, 0, 0) * kNetC + c * 8 : 0), in);
    }
    for (int i = threadIdx.x; i < NZR * RH * RW; i += blockDim.x) {
      const int px = i % RW, row = (i / RW) % RH, dz = i / (RW * RH);
      const int xx = min(max(x0 + px - 1, 0), sh.nx - 1), yy = min(max(y0 + row - 1, 0), sh.ny - 1);
      const int zz = NDIM == 3 ? min(max(z + dz - 1, 0), sh.nz - 1) : 0;
      cp_async4(tp + (dz * RH + row) * kEndRow1 + px, phi + sh.u(b, zz, yy, xx), true);
    }
    cp_async_wait();
    __syncthreads();
    const int row = 2 * (warp & 3) + (lane >> 4), xs = 16 * (warp >> 2);
    const unsigned char *pg = tg + (row * kEndRow + xs) * 64 + (lane & 15) * 4;
    const float *pp = tp + row * kEndRow1 + xs;
#pragma unroll(NDIM == 3 ? 2 : 16)
    for (int i = 0; i < 16; ++i) {
      const float2 gf = ld_bf2(pg + i * 64);  // (zero outside the grid)
      const uint64_t g = pack2(gf.x, gf.y);
      db = add2(db, g);
#pragma unroll
      for (int t = 0; t < T; ++t) {
        const int ox = t % 3, oy = (t / 3) % 3, dz = t / 9;
        const float p = pp[(dz * RH + oy) * kEndRow1 + i + ox];
        dw[t] = fma2(pack2(p, p), g, dw[t]);
      }
    }
  }
  __syncthreads();
  end_reduce<T>(acc, dw, grads + gw_off);
  __syncthreads();
  end_reduce<1>(acc, &db, grads + gb_off);
}

// ---------------------------------------------------------- optimiser -----
__global__ void net_adam_k(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                           float *__restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                           float c1, float c2) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
  }
}

// BF16 B operands of the four 32 -> 32 layers: forward Wf[l][co][t][ci] =
// W[t][ci][co] and data gradient Wd[l][ci][t][co] = W[T-1-t][ci][co] (taps
// mirrored: the transposed convolution reads p - t).
__global__ void net_pack_k(const float *__restrict__ params, int T, int64_t w0, int64_t w1,
                           int64_t w2, int64_t w3, bf16 *__restrict__ wf, bf16 *__restrict__ wd) {
  const int64_t per = (int64_t)kNetC * T * kNetC;
  const int64_t total = 4 * per;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int l = (int)(i / per);
    int64_t r = i % per;
    const int c = (int)(r % kNetC);
    r /= kNetC;
    const int t = (int)(r % T);
    const int nrow = (int)(r / T);
    const int64_t woff = l == 0 ? w0 : l == 1 ? w1 : l == 2 ? w2 : w3;
    // forward: row n = co, column (t, ci = c)
    wf[i] = __float2bfloat16_rn(params[woff + ((int64_t)t * kNetC + c) * kNetC + nrow]);
    // data gradient: row n = ci, column (t, co = c) from tap T-1-t
    wd[i] = __float2bfloat16_rn(params[woff + ((int64_t)(T - 1 - t) * kNetC + nrow) * kNetC + c]);
  }
}

// ------------------------------------------------------------ launchers ----
// Dynamic shared-memory limits of the kernels that need more than the
// default, once per device (thread-safe; the occupancy query is unused).
template <int NDIM>
static cudaError_t setup_attrs() {
  static KernelSetup k_last_t, k_last_f, k_faces;
  int occ = 0;
  cudaError_t e;
  e = kernel_setup(k_last_t, (const void *)net_last_fwd_k<NDIM, true>, 32, last_smem_bytes<NDIM>(), &occ);
  if (e != cudaSuccess) return e;
  e = kernel_setup(k_last_f, (const void *)net_last_fwd_k<NDIM, false>, 32, last_smem_bytes<NDIM>(), &occ);
  if (e != cudaSuccess) return e;
  return kernel_setup(k_faces, (const void *)net_dgrad_faces_k<NDIM>, 32,
                      faces_smem<NDIM>(), &occ);
}

template <int NDIM>
static cudaError_t net_forward_t(const NetBuffers &nb, const NetShape &sh, const float *phi,
                                 float scale, float *phihat, const float *target, bool train,
                                 int num_sms, cudaStream_t s) {
  cudaError_t e = setup_attrs<NDIM>();
  if (e != cudaSuccess) return e;
  const NetLayout &L = nb.layout;
  // 32-bit tile and pixel indices, here as in the convolutions
  if (sh.padded_cells() >= (int64_t)INT32_MAX) return cudaErrorInvalidValue;
  const int64_t first_tiles = (int64_t)sh.batch * sh.nz * ((sh.nx + 31) / 32) * ((sh.ny + 7) / 8);
  const int first_grid = (int)std::min<int64_t>(
      first_tiles, (int64_t)num_sms * (train ? first_blocks<NDIM, true>() : first_blocks<NDIM, false>()));
  if (train)
    net_first_fwd_k<NDIM, true><<<first_grid, 256, 0, s>>>(phi, nb.params, L.w[0], L.b[0], sh, nb.z[0], nb.a[0]);
  else
    net_first_fwd_k<NDIM, false><<<first_grid, 256, 0, s>>>(phi, nb.params, L.w[0], L.b[0], sh, nullptr, nb.a[0]);
  const int64_t per = (int64_t)kNetC * net_taps(NDIM) * kNetC;
  for (int l = 1; l <= 4; ++l) {
    bf16 *in = nb.a[(l - 1) % (train ? 5 : 2)];
    bf16 *out = nb.a[l % (train ? 5 : 2)];
    e = net_conv_rows(0, in, nb.wf + (l - 1) * per, nb.params + L.b[l], sh,
                      train ? nb.z[l] : nullptr, out, nullptr, nullptr, nb.status, num_sms, s);
    if (e != cudaSuccess) return e;
  }
  const bf16 *a5 = nb.a[4 % (train ? 5 : 2)];
  const int64_t last_items = (int64_t)sh.batch * sh.nz * ((sh.ny + kLastTY - 1) / kLastTY) *
                             ((sh.nx + kLastTX - 1) / kLastTX);
  const int last_grid = (int)std::min<int64_t>(last_items, (int64_t)num_sms * 2);
  if (train)
    net_last_fwd_k<NDIM, true><<<last_grid, 256, last_smem_bytes<NDIM>(), s>>>(a5, nb.params, L.w[5], L.b[5], sh, phi, scale, phihat, target, nb.g6, nb.loss);
  else
    net_last_fwd_k<NDIM, false><<<last_grid, 256, last_smem_bytes<NDIM>(), s>>>(a5, nb.params, L.w[5], L.b[5], sh, phi, scale, phihat, nullptr, nullptr, nullptr);
  return cudaGetLastError();
}

template <int NDIM>
static cudaError_t net_backward_t(const NetBuffers &nb, const NetShape &sh, const float *phi,
                                  int num_sms, cudaStream_t s) {
  const NetLayout &L = nb.layout;
  const int64_t n = sh.cells();
  static KernelSetup k_last, k_first;
  int occ_last = 1, occ_first = 1;
  cudaError_t e = kernel_setup(k_last, (const void *)net_last_bwd_k<NDIM>, 256, last_bwd_smem<NDIM>(), &occ_last);
  if (e != cudaSuccess) return e;
  e = kernel_setup(k_first, (const void *)net_first_wgrad_k<NDIM>, 256, first_wgrad_smem<NDIM>(), &occ_first);
  if (e != cudaSuccess) return e;
  const int64_t end_items = (int64_t)sh.batch * sh.nz * ((sh.ny + kEndTY - 1) / kEndTY) *
                            ((sh.nx + kEndTX - 1) / kEndTX);
  net_last_bwd_k<NDIM><<<(int)std::min<int64_t>(end_items, (int64_t)num_sms * occ_last), 256,
                         last_bwd_smem<NDIM>(), s>>>(nb.g6, nb.params, L.w[5], sh, nb.z[4], nb.a[4], nb.gz[4],
                                                     nb.grads, L.w[5], L.b[5]);
  const int64_t per = (int64_t)kNetC * net_taps(NDIM) * kNetC;
  for (int l = 4; l >= 1; --l) {
    e = net_wgrad(nb.a[l - 1], nb.gz[l], sh, nb.grads + L.w[l], nb.grads + L.b[l], nb.status,
                              num_sms, s);
    if (e != cudaSuccess) return e;
    e = net_conv_rows(1, nb.gz[l], nb.wd + (l - 1) * per, nullptr, sh, nullptr, nb.gz[l - 1], nb.raw,
                      nb.z[l - 1], nb.status, num_sms, s);
    if (e != cudaSuccess) return e;
    net_dgrad_faces_k<NDIM><<<(int)std::min<int64_t>((n + kFacesThreads / 32 - 1) / (kFacesThreads / 32), (int64_t)num_sms * (NDIM == 3 ? 1 : 2)), kFacesThreads, faces_smem<NDIM>(), s>>>(
        nb.raw, nb.gz[l], nb.params, L.w[l], sh, nb.z[l - 1], nb.gz[l - 1]);
  }
  net_first_wgrad_k<NDIM><<<(int)std::min<int64_t>(end_items, (int64_t)num_sms * occ_first), 256,
                            first_wgrad_smem<NDIM>(), s>>>(phi, nb.gz[0], sh, nb.grads, L.w[0], L.b[0]);
  return cudaGetLastError();
}

cudaError_t net_forward(const NetBuffers &nb, const NetShape &sh, const float *phi, float scale,
                        float *phihat, const float *target, bool train, int num_sms, cudaStream_t s) {
  return sh.ndim == 3 ? net_forward_t<3>(nb, sh, phi, scale, phihat, target, train, num_sms, s)
                      : net_forward_t<2>(nb, sh, phi, scale, phihat, target, train, num_sms, s);
}

cudaError_t net_backward(const NetBuffers &nb, const NetShape &sh, const float *phi, int num_sms,
                         cudaStream_t s) {
  return sh.ndim == 3 ? net_backward_t<3>(nb, sh, phi, num_sms, s) : net_backward_t<2>(nb, sh, phi, num_sms, s);
}

cudaError_t net_pack(const NetBuffers &nb, cudaStream_t s) {
  const NetLayout &L = nb.layout;
  net_pack_k<<<256, 256, 0, s>>>(nb.params, L.T, L.w[1], L.w[2], L.w[3], L.w[4], nb.wf, nb.wd);
  return cudaGetLastError();
}

cudaError_t net_adam(const NetBuffers &nb, float lr, float b1, float b2, float eps, int step,
                     cudaStream_t s) {
  const float c1 = 1.0f / (1.0f - powf(b1, (float)step));
  const float c2 = 1.0f / (1.0f - powf(b2, (float)step));
  net_adam_k<<<256, 256, 0, s>>>(nb.params, nb.grads, nb.m, nb.v, nb.layout.total, lr, b1, b2, eps, c1, c2);
  return net_pack(nb, s);
}

}  // namespace ac
