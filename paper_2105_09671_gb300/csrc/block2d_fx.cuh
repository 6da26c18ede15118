// 2D register-tile stencil with temporal blocking for FP64 grids of modest
// size (integer form of the update, fixed64.cuh).
//
// As block2d.cuh with one cell per lane and row: a CTA owns 32 columns x
// (warps x R) rows, advances them k steps between one load and one store, and
// writes the tile less k cells per side.  Small grids are bound by the latency
// of a launch and of a cell's chain of ~100 dependent instructions, which a
// launch of several steps pays once and R rows and several warps overlap.
#pragma once

#include "fixed64.cuh"
#include "kernels.h"

namespace ac {

constexpr int kB2FxMaxWarps = 16;
// first and last row of each warp, by step parity: m, value, exponent
constexpr int b2fx_smem_bytes(int warps) { return 4 * warps * 32 * 20; }

template <int R>
__global__ void __launch_bounds__(kB2FxMaxWarps * 32)
    block2d_fx_k(const double *__restrict__ src, double *__restrict__ dst, GridParams g, int k) {
  extern __shared__ __align__(16) unsigned char fsm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  // [step parity][first, last row][warp][lane]
  int64_t *sm = reinterpret_cast<int64_t *>(fsm);
  double *sv = reinterpret_cast<double *>(sm + 4 * nw * 32);
  int *se = reinterpret_cast<int *>(sv + 4 * nw * 32);
  const int nx = (int)g.nx, ny = (int)g.ny;
  const int x0 = (int)blockIdx.x * (32 - 2 * k) - k, y0 = (int)blockIdx.y * (nw * R - 2 * k) - k;
  const int x = x0 + lane, yr = y0 + warp * R;
  const Coef<double> coef(g);
  // The previous launch on the stream writes what this one reads.
  pdl_wait();
  double v[R];
  FxV f[R];
  const int xi = reflect(x, nx);
#pragma unroll
  for (int r = 0; r < R; ++r) {
    v[r] = src[(int64_t)reflect(yr + r, ny) * g.pitch + xi];
    f[r] = fx_in(v[r], coef.limit);
  }
  for (int s = 0; s < k; ++s) {
    const int first = (s & 1) * 2 * nw * 32 + lane, last = first + nw * 32;
    sm[first + warp * 32] = f[0].m;
    sv[first + warp * 32] = v[0];
    se[first + warp * 32] = f[0].e;
    sm[last + warp * 32] = f[R - 1].m;
    sv[last + warp * 32] = v[R - 1];
    se[last + warp * 32] = f[R - 1].e;
    __syncthreads();
    const int ib = last + max(warp - 1, 0) * 32, ia = first + min(warp + 1, nw - 1) * 32;
    FxV lo, hi;
    lo.m = sm[ib];
    lo.e = se[ib];
    hi.m = sm[ia];
    hi.e = se[ia];
    double nv[R];
    uint32_t fp64 = 0;  // rows whose cell takes the FP64 operations
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const FxV w = fx_shfl<-1>(f[r]), ea = fx_shfl<1>(f[r]);
      const FxV &b = r == 0 ? lo : f[r > 0 ? r - 1 : 0], &a = r == R - 1 ? hi : f[r + 1 < R ? r + 1 : 0];
      const int m = max(max(max(w.e, ea.e), max(b.e, a.e)), f[r].e);
      const int64_t ns = (fx_align(w, m) + fx_align(ea, m)) + (fx_align(b, m) + fx_align(a, m));
      if (!fx_update<2>(f[r], ns, m, coef, &nv[r])) fp64 |= 1u << r;
    }
    const uint32_t any = __reduce_or_sync(0xffffffffu, fp64);
    if (any) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!((any >> r) & 1u)) continue;
        const double vw = __shfl_up_sync(0xffffffffu, v[r], 1), ve = __shfl_down_sync(0xffffffffu, v[r], 1);
        const double vb = r == 0 ? sv[ib] : v[r > 0 ? r - 1 : 0], va = r == R - 1 ? sv[ia] : v[r + 1 < R ? r + 1 : 0];
        if ((fp64 >> r) & 1u) nv[r] = fx_plain<2>(v[r], {vw, ve, vb, va}, coef);
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      v[r] = nv[r];
      f[r] = fx_in(nv[r], coef.limit);
    }
  }
  pdl_launch_dependents();
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int tr = warp * R + r, y = yr + r;
    if (tr >= k && tr < nw * R - k && y < ny && lane >= k && lane < 32 - k && x < nx)
      dst[(int64_t)y * g.pitch + x] = v[r];
  }
}

}  // namespace ac
