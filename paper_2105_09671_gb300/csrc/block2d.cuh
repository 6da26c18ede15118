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
// is one to two instructions per cell and step, against 3.9 (8-cell strips) to
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

  // Rows live in R + 1 slots.  An ascending step finds row r in slot r + 1 and
  // leaves it in slot r, a descending one moves it back: the slot written is
  // that of a row no longer needed, so an update in place costs no register
  // moves (1.4 of 11.4 instructions an update before).  The free slot takes
  // the neighbour warp's row.
  float v[R + 1][E];
  if (x0 >= 0 && x0 + 32 * E <= nx && y0 >= 0 && y0 + nw * R <= ny) {
    const T *p = src + (int64_t)yr * g.pitch + xl;
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int q = 0; q < E / V; ++q) ld_cells<T, V>(p + (int64_t)r * g.pitch + q * V, v[r + 1] + q * V);
  } else {
    int xi[E];
#pragma unroll
    for (int e = 0; e < E; ++e) xi[e] = reflect(xl + e, nx);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const T *p = src + (int64_t)reflect(yr + r, ny) * g.pitch;
#pragma unroll
      for (int e = 0; e < E; ++e) v[r + 1][e] = to_c(p[xi[e]]);
    }
  }

  // Each warp publishes its first and last row; two buffers by step parity,
  // so one barrier per step orders both the reads and the next writes.  The
  // tile's outermost rows and columns see a wrong neighbour (their own value
  // or a neighbour lane's); the error moves inwards one cell per step and
  // stays in the halo.
  const int ws = 32 * E;
  auto put = [](float *p, const float *a) {
#pragma unroll
    for (int q = 0; q < E / 4; ++q)
      *reinterpret_cast<float4 *>(p + q * 128) = make_float4(a[4 * q], a[4 * q + 1], a[4 * q + 2], a[4 * q + 3]);
  };
  auto get = [](const float *p, float *a) {
#pragma unroll
    for (int q = 0; q < E / 4; ++q) {
      const float4 f = *reinterpret_cast<const float4 *>(p + q * 128);
      a[4 * q] = f.x; a[4 * q + 1] = f.y; a[4 * q + 2] = f.z; a[4 * q + 3] = f.w;
    }
  };
  float *const my = edge + warp * ws + lane * 4;
  const int to_below = ((warp > 0 ? nw - 1 : nw)) * ws, to_above = warp + 1 < nw ? ws : 0;  // from my
  auto step = [&]<bool UP>(int s) {
    constexpr int O = UP ? 1 : 0;  // row r is in slot r + O before the step
    float *buf = my + (UP ? 0 : 2 * nw * ws);
    put(buf, v[O]);
    put(buf + nw * ws, v[R - 1 + O]);
    __syncthreads();
    float far[E];  // the outer row of the row formed last
    get(buf + to_below, UP ? v[0] : far);
    get(buf + to_above, UP ? far : v[R]);
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int r = UP ? q : R - 1 - q;
      const float *cur = v[r + O];
      float *out = v[r + 1 - O];                      // the row before it in this step's order
      const float *next = q == R - 1 ? far : v[UP ? (r + 2 <= R ? r + 2 : R) : (r > 0 ? r - 1 : 0)];
      const float left = __shfl_up_sync(0xffffffffu, cur[E - 1], 1);
      const float right = __shfl_down_sync(0xffffffffu, cur[0], 1);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const float w = e == 0 ? left : cur[e - 1];
        const float ea = e == E - 1 ? right : cur[e + 1];
        out[e] = ac_update<float>(cur[e], (w + ea) + (out[e] + next[e]), -4.0f, alpha, beta);
      }
    }
    if constexpr (sizeof(T) == 2) {
      if ((round_mask >> s) & 1u) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int e = 0; e < E; ++e) v[r + 1 - O][e] = to_c(from_c<T>(v[r + 1 - O][e]));
      }
    }
  };
  int s = 0;
  for (; s + 2 <= k; s += 2) {
    step.template operator()<true>(s);
    step.template operator()<false>(s + 1);
  }
  if (s < k) step.template operator()<true>(s);

  // The next launch's CTAs may take an SM once this grid's have all come
  // here.  (Let in at the start they settle beside CTAs that still step, two
  // to an SM while others idle: 512^2 0.67 us a step against 0.50.)
  pdl_launch_dependents();
  const int rlo = k, rhi = nw * R - k;  // output rows of the tile
  auto store = [&]<int O>() {
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
          st_cells<T, V>(p + x, v[r + O] + q * V);
        } else {
#pragma unroll
          for (int e = 0; e < V; ++e)
            if (x + e < nx) p[x + e] = from_c<T>(v[r + O][q * V + e]);
        }
      }
    }
  };
  if (k % 2) store.template operator()<0>();
  else store.template operator()<1>();
}

}  // namespace ac
