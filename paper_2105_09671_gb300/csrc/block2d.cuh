// 2D register-tile stencil with temporal blocking: the default schedule's
// kernel for FP32 and FP16 storage.
//
// One CTA owns a tile of 32 E columns x (warps x R) rows, held in registers:
// a lane owns E adjacent cells of R adjacent rows.  The tile is loaded once,
// advanced k steps, and its interior (the tile less a halo of hx >= k
// columns and k rows per side) is written.
//
// Per step and row a warp issues two shuffles (the x neighbours across
// lanes) and the update's 8 FP32 operations per cell; the rows above and
// below a warp's own come through shared memory, one CTA barrier per step.
// Boundary cells cost nothing: see reflect() in common.cuh.  Beside the 8 operations that
// is about 0.8 instructions per cell and step, against 3.9 (8-cell strips) to
// 7.1 in the streaming kernel, and a step's latency is one tile step (0.17 us)
// where a pass of the streaming kernel walks a chunk of rows one by one.
#pragma once

#include <cmath>

#include "kernels.h"

namespace ac {

constexpr int kB2MaxWarps = 16;
constexpr int b2_smem_bytes(int E, int warps) { return 4 * warps * 32 * E * (int)sizeof(float); }

// MINB: CTAs of kB2MaxWarps warps per SM that the register budget allows.
// round_mask bit s: the values are rounded to the storage type after step
// s + 1 (FP16 storage: where a pass of the schedule ends inside a launch).
template <typename T, int E, int R, int MINB>
__global__ void __launch_bounds__(kB2MaxWarps * 32, MINB)
    block2d_k(const T *__restrict__ src, T *__restrict__ dst, GridParams g, int k, int hx,
              uint32_t round_mask) {
  static_assert(sizeof(typename Traits<T>::C) == 4, "FP32 arithmetic");
  constexpr int V = Traits<T>::V < E ? Traits<T>::V : E;  // cells per memory vector (16 or 8 bytes)
  static_assert(E % 4 == 0 && E % V == 0, "whole vectors per lane");
  extern __shared__ __align__(16) float edge[];  // [step parity][first, last row][warp][E/4][32][4]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int nx = (int)g.nx, ny = (int)g.ny;
  const int x0 = (int)blockIdx.x * (32 * E - 2 * hx) - hx;
  const int y0 = (int)blockIdx.y * (nw * R - 2 * k) - k;
  const int xl = x0 + lane * E, yr = y0 + warp * R;
  const float alpha = (float)g.alpha, beta = (float)g.beta;
  // The previous launch on the stream writes what this one reads.
  pdl_wait();

  float v[R][E];
  if (x0 >= 0 && x0 + 32 * E <= nx && y0 >= 0 && y0 + nw * R <= ny) {
    const T *p = src + (int64_t)yr * g.pitch + xl;
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int q = 0; q < E / V; ++q) ld_cells<T, V>(p + (int64_t)r * g.pitch + q * V, v[r] + q * V);
  } else {
    int xi[E];
#pragma unroll
    for (int e = 0; e < E; ++e) xi[e] = reflect(xl + e, nx);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const T *p = src + (int64_t)reflect(yr + r, ny) * g.pitch;
#pragma unroll
      for (int e = 0; e < E; ++e) v[r][e] = to_c(p[xi[e]]);
    }
  }

  // Each warp publishes its first and last row; two buffers by step parity,
  // so one barrier per step orders both the reads and the next writes.  The
  // tile's outermost rows and columns see a wrong neighbour (their own value
  // or a neighbour lane's); the error moves inwards one cell per step and
  // stays in the halo.
  const int ws = 32 * E;
  for (int s = 0; s < k; ++s) {
    float *first = edge + (s & 1) * 2 * nw * ws + lane * 4, *last = first + nw * ws;
#pragma unroll
    for (int q = 0; q < E / 4; ++q) {
      *reinterpret_cast<float4 *>(first + warp * ws + q * 128) =
          make_float4(v[0][4 * q], v[0][4 * q + 1], v[0][4 * q + 2], v[0][4 * q + 3]);
      *reinterpret_cast<float4 *>(last + warp * ws + q * 128) =
          make_float4(v[R - 1][4 * q], v[R - 1][4 * q + 1], v[R - 1][4 * q + 2], v[R - 1][4 * q + 3]);
    }
    __syncthreads();
    const float *pb = last + max(warp - 1, 0) * ws, *pa = first + min(warp + 1, nw - 1) * ws;
    float prev[E], above[E];
#pragma unroll
    for (int q = 0; q < E / 4; ++q) {
      const float4 b = *reinterpret_cast<const float4 *>(pb + q * 128);
      const float4 a = *reinterpret_cast<const float4 *>(pa + q * 128);
      prev[4 * q] = b.x; prev[4 * q + 1] = b.y; prev[4 * q + 2] = b.z; prev[4 * q + 3] = b.w;
      above[4 * q] = a.x; above[4 * q + 1] = a.y; above[4 * q + 2] = a.z; above[4 * q + 3] = a.w;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float cur[E];
#pragma unroll
      for (int e = 0; e < E; ++e) cur[e] = v[r][e];
      const float left = __shfl_up_sync(0xffffffffu, cur[E - 1], 1);
      const float right = __shfl_down_sync(0xffffffffu, cur[0], 1);
      float out[E];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const float w = e == 0 ? left : cur[e - 1];
        const float ea = e == E - 1 ? right : cur[e + 1];
        const float nn = r == R - 1 ? above[e] : v[r + 1 < R ? r + 1 : 0][e];
        out[e] = ac_update<float>(cur[e], (w + ea) + (prev[e] + nn), -4.0f, alpha, beta);
      }
#pragma unroll
      for (int e = 0; e < E; ++e) v[r][e] = out[e];
#pragma unroll
      for (int e = 0; e < E; ++e) prev[e] = cur[e];
    }
    if constexpr (sizeof(T) == 2) {
      if ((round_mask >> s) & 1u) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int e = 0; e < E; ++e) v[r][e] = to_c(from_c<T>(v[r][e]));
      }
    }
  }

  // The next launch's CTAs may take an SM once this grid's have all come
  // here.  (Let in at the start they settle beside CTAs that still step, two
  // to an SM while others idle: 512^2 0.67 us a step against 0.50.)
  pdl_launch_dependents();
  const int rlo = k, rhi = nw * R - k;  // output rows of the tile
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int tr = warp * R + r, y = yr + r;
    if (tr < rlo || tr >= rhi || y >= ny) continue;
    T *p = dst + (int64_t)y * g.pitch;
#pragma unroll
    for (int q = 0; q < E / V; ++q) {
      const int c = lane * E + q * V, x = x0 + c;
      if (c < hx || c >= 32 * E - hx || x >= nx) continue;
      if (x + V <= nx) {
        st_cells<T, V>(p + x, v[r] + q * V);
      } else {
#pragma unroll
        for (int e = 0; e < V; ++e)
          if (x + e < nx) p[x + e] = from_c<T>(v[r][q * V + e]);
      }
    }
  }
}

}  // namespace ac
