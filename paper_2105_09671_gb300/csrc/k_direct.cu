// Direct stencil kernels: one explicit Euler step (Eq. pytorchACeq) per
// launch, every neighbour read from global memory with its index clamped to
// the domain, which realises the zero-Neumann ghost copy of Section 2
// (the ghost equals its adjacent interior cell).  This is the plain variant
// the streaming kernels are checked and timed against.
//
// Larger FP64 grids march: a value is taken apart for the integer form of the
// update (fixed64.cuh) once per lane and shared by warp shuffles (x) and
// registers (y, z) while a warp walks a chunk of rows or planes.
#include <algorithm>

#include "fixed64.cuh"
#include "kernels.h"

namespace ac {

template <typename T>
__device__ __forceinline__ void step2d_cell(const T *__restrict__ src, T *__restrict__ dst,
                                            const GridParams &g, int64_t i, int64_t j) {
  using C = typename Traits<T>::C;
  const int64_t im = i > 0 ? i - 1 : 0, ip = i + 1 < g.nx ? i + 1 : i;
  const int64_t jm = j > 0 ? j - 1 : 0, jp = j + 1 < g.ny ? j + 1 : j;
  const T *row = src + j * g.pitch;
  C p = to_c(row[i]);
  C w = to_c(row[im]), e = to_c(row[ip]);
  C s = to_c(src[jm * g.pitch + i]), n = to_c(src[jp * g.pitch + i]);
  const Coef<C> c(g);
  if constexpr (sizeof(T) == 8) dst[j * g.pitch + i] = fx_cell<2>(p, {w, e, s, n}, c);
  else dst[j * g.pitch + i] = from_c<T>(ac_update<C>(p, (w + e) + (s + n), C(-4), c.alpha, c.beta));
}

template <typename T>
__device__ __forceinline__ void step3d_cell(const T *__restrict__ src, T *__restrict__ dst,
                                            const GridParams &g, int64_t i, int64_t j, int64_t k) {
  using C = typename Traits<T>::C;
  const int64_t im = i > 0 ? i - 1 : 0, ip = i + 1 < g.nx ? i + 1 : i;
  const int64_t jm = j > 0 ? j - 1 : 0, jp = j + 1 < g.ny ? j + 1 : j;
  const int64_t km = k > 0 ? k - 1 : 0, kp = k + 1 < g.nz ? k + 1 : k;
  const int64_t plane = g.pitch * g.ny;
  const T *row = src + k * plane + j * g.pitch;
  C p = to_c(row[i]);
  C w = to_c(row[im]), e = to_c(row[ip]);
  C s = to_c(src[k * plane + jm * g.pitch + i]), n = to_c(src[k * plane + jp * g.pitch + i]);
  C b = to_c(src[km * plane + j * g.pitch + i]), f = to_c(src[kp * plane + j * g.pitch + i]);
  const Coef<C> c(g);
  if constexpr (sizeof(T) == 8) dst[k * plane + j * g.pitch + i] = fx_cell<3>(p, {w, e, s, n, b, f}, c);
  else dst[k * plane + j * g.pitch + i] =
      from_c<T>(ac_update<C>(p, ((w + e) + (s + n)) + (b + f), C(-6), c.alpha, c.beta));
}

// one thread per x; y and z as for_cell_yz (see cell_grid)
template <typename T, bool TALL>
__global__ void __launch_bounds__(256) step2d_direct(const T *__restrict__ src,
                                                     T *__restrict__ dst, GridParams g) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_wait();  // (see direct_t)
  pdl_launch_dependents();
  if (i >= g.nx) return;
  for_cell_yz<TALL>(g, [&](int64_t j, int64_t) { step2d_cell(src, dst, g, i, j); });
}

template <typename T, bool TALL>
__global__ void __launch_bounds__(256) step3d_direct(const T *__restrict__ src,
                                                     T *__restrict__ dst, GridParams g) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_wait();  // (see direct_t)
  pdl_launch_dependents();
  if (i >= g.nx) return;
  for_cell_yz<TALL>(g, [&](int64_t j, int64_t k) { step3d_cell(src, dst, g, i, j, k); });
}

// -------------------------------------------------- FP64, integer form --
// Grids that march.  Below, a march's few warps wait for one row (plane) after
// another: one thread a cell takes 3.8 us a step against 4.9 at 512^2, 4.5
// against 7.9 at 64^3 and 9.5 against 10.3 at 80^3; 10.5 against 10.3 at 1024^2,
// 16.2 against 15.1 at 100^3.  In 3D rows that fill its blocks move the line up
// (128^3 25.8 against 29.4; 256^3 197 against 164).
static bool fx_marches(int ndim, const GridParams &g) {
  const int64_t cells = g.nx * g.ny * g.nz;
  if (ndim == 2) return cells >= 1000000;
  const int64_t full = (g.nx + kCellBlockX - 1) / kCellBlockX * kCellBlockX * g.ny * g.nz;
  return cells >= (10 * full <= 11 * cells ? 3000000 : 700000);
}
constexpr int kFxWarps = 4;                      // per CTA, independent of one another
constexpr int kFx2E = 4, kFx2W = 32 * kFx2E;      // 2D: cells a lane, columns a warp
constexpr int kFx3E = 2, kFx3W = 32 * kFx3E;      // 3D
constexpr int kFx3R = 2;                         // 3D: rows a warp writes per plane
constexpr int kFxHalo = 2;                       // halo columns per side (one 16-byte vector)

// One row's cells of a lane: E cells from column xl, or from the reflected
// columns xi where the strip leaves the grid.
template <int E>
__device__ __forceinline__ void fx_load(const double *row, int xl, const int *xi, bool inside, double *v) {
  if (inside) {
#pragma unroll
    for (int q = 0; q < E; q += 2) {
      const double2 d = *reinterpret_cast<const double2 *>(row + xl + q);
      v[q] = d.x;
      v[q + 1] = d.y;
    }
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = row[xi[e]];
  }
}
// Store of the cells that are outputs of the strip (columns kFxHalo .. W - kFxHalo) and in the grid.
template <int E>
__device__ __forceinline__ void fx_store(double *row, int xl, int lane, int nx, const double *v) {
#pragma unroll
  for (int q = 0; q < E; q += 2) {
    const int c = lane * E + q, x = xl + q;
    if (c < kFxHalo || c >= 32 * E - kFxHalo || x >= nx) continue;
    if (x + 1 < nx) *reinterpret_cast<double2 *>(row + x) = make_double2(v[q], v[q + 1]);
    else row[x] = v[q];
  }
}

// A warp owns kFx2W columns and marches over `chunk` rows.  Bound by integer
// issue (some 164 instructions a cell, 14 of them wide multiply-adds, which
// take more than one slot: 64 % of the slots busy): 4096^2 253 -> 104 us a
// step (from noise 113: more cells take the FP64 operations), 2048^2 64 -> 30
// against the FP64 operations alone.
__global__ void __launch_bounds__(kFxWarps * 32, 6) step2d_fx(const double *__restrict__ src,
                                                           double *__restrict__ dst, GridParams g, int strips,
                                                           int chunk) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = (int64_t)blockIdx.x * kFxWarps + (threadIdx.x >> 5);
  const int nx = (int)g.nx, ny = (int)g.ny;
  const int x0 = (int)(gw % strips) * (kFx2W - 2 * kFxHalo) - kFxHalo, xl = x0 + lane * kFx2E;
  const int64_t ys = gw / strips * chunk;
  if (ys >= ny) return;
  const int ya = (int)ys, ye = min(ny, ya + chunk);
  const bool inside = x0 >= 0 && x0 + kFx2W <= nx;
  int xi[kFx2E];
#pragma unroll
  for (int e = 0; e < kFx2E; ++e) xi[e] = reflect(xl + e, nx);
  const Coef<double> coef(g);
  double v[kFx2E];
  FxV below[kFx2E], x[kFx2E];  // the row below, the row
  fx_load<kFx2E>(src + (int64_t)reflect(ya - 1, ny) * g.pitch, xl, xi, inside, v);
#pragma unroll
  for (int e = 0; e < kFx2E; ++e) below[e] = fx_in(v[e], coef.limit);
  fx_load<kFx2E>(src + (int64_t)ya * g.pitch, xl, xi, inside, v);
#pragma unroll
  for (int e = 0; e < kFx2E; ++e) x[e] = fx_in(v[e], coef.limit);
  fx_load<kFx2E>(src + (int64_t)reflect(ya + 1, ny) * g.pitch, xl, xi, inside, v);
  for (int y = ya; y < ye; ++y) {
    FxV up[kFx2E];
#pragma unroll
    for (int e = 0; e < kFx2E; ++e) up[e] = fx_in(v[e], coef.limit);
    if (y + 1 < ye)  // the row after next, ahead of its use
      fx_load<kFx2E>(src + (int64_t)reflect(y + 2, ny) * g.pitch, xl, xi, inside, v);
    const FxV left = fx_shfl<-1>(x[kFx2E - 1]), right = fx_shfl<1>(x[0]);
    double out[kFx2E];
    bool ok[kFx2E], all = true;
#pragma unroll
    for (int e = 0; e < kFx2E; ++e) {
      const FxV &w = e == 0 ? left : x[e - 1], &ea = e == kFx2E - 1 ? right : x[e + 1];
      const int m = max(max(max(w.e, ea.e), max(below[e].e, up[e].e)), x[e].e);
      const int64_t ns = (fx_align(w, m) + fx_align(ea, m)) + (fx_align(below[e], m) + fx_align(up[e], m));
      ok[e] = fx_update<2>(x[e], ns, m, coef, &out[e]);
      all = all && ok[e];
    }
    if (!all) {  // some take the FP64 operations, from memory
      const double *row = src + (int64_t)y * g.pitch;
      const double *rs = src + (int64_t)max(y - 1, 0) * g.pitch, *rn = src + (int64_t)min(y + 1, ny - 1) * g.pitch;
#pragma unroll
      for (int e = 0; e < kFx2E; ++e) {
        if (ok[e]) continue;
        const int im = xi[e] > 0 ? xi[e] - 1 : 0, ip = min(xi[e] + 1, nx - 1);
        out[e] = fx_plain<2>(row[xi[e]], {row[im], row[ip], rs[xi[e]], rn[xi[e]]}, coef);
      }
    }
    fx_store<kFx2E>(dst + (int64_t)y * g.pitch, xl, lane, nx, out);
#pragma unroll
    for (int e = 0; e < kFx2E; ++e) {
      below[e] = x[e];
      x[e] = up[e];
    }
  }
}

// A warp owns kFx3W columns of kFx3R rows and marches over `chunk` planes; it
// takes apart kFx3R + 2 rows of each plane (against a barrier a plane to share
// them; two rows in 128 registers rather than three or four in 160).  256^3
// 317 -> 165 us a step, 200 x 100 x 100 45 -> 27.
__global__ void __launch_bounds__(kFxWarps * 32) step3d_fx(const double *__restrict__ src,
                                                           double *__restrict__ dst, GridParams g, int strips,
                                                           int bands, int chunk) {
  constexpr int R = kFx3R, E = kFx3E;
  const int lane = threadIdx.x & 31;
  const int64_t gw = (int64_t)blockIdx.x * kFxWarps + (threadIdx.x >> 5);
  const int nx = (int)g.nx, ny = (int)g.ny, nz = (int)g.nz;
  const int x0 = (int)(gw % strips) * (kFx3W - 2 * kFxHalo) - kFxHalo, xl = x0 + lane * E;
  const int y0 = (int)(gw / strips % bands) * R;
  const int64_t zs = gw / strips / bands * chunk;
  if (zs >= nz) return;
  const int za = (int)zs, ze = min(nz, za + chunk);
  const int64_t plane = g.pitch * g.ny;
  const bool inside = x0 >= 0 && x0 + kFx3W <= nx;
  int xi[E];
#pragma unroll
  for (int e = 0; e < E; ++e) xi[e] = reflect(xl + e, nx);
  int64_t ro[R + 2];
#pragma unroll
  for (int r = 0; r < R + 2; ++r) ro[r] = (int64_t)reflect(y0 - 1 + r, ny) * g.pitch;
  const Coef<double> coef(g);
  FxV below[R][E], x[R + 2][E];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    double v[E];
    fx_load<E>(src + (int64_t)reflect(za - 1, nz) * plane + ro[r + 1], xl, xi, inside, v);
#pragma unroll
    for (int e = 0; e < E; ++e) below[r][e] = fx_in(v[e], coef.limit);
  }
#pragma unroll
  for (int r = 0; r < R + 2; ++r) {
    double v[E];
    fx_load<E>(src + (int64_t)za * plane + ro[r], xl, xi, inside, v);
#pragma unroll
    for (int e = 0; e < E; ++e) x[r][e] = fx_in(v[e], coef.limit);
  }
  for (int z = za; z < ze; ++z) {
    FxV up[R + 2][E];
    const double *zp = src + (int64_t)reflect(z + 1, nz) * plane;
#pragma unroll
    for (int r = 0; r < R + 2; ++r) {
      double v[E];
      fx_load<E>(zp + ro[r], xl, xi, inside, v);
#pragma unroll
      for (int e = 0; e < E; ++e) up[r][e] = fx_in(v[e], coef.limit);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const FxV left = fx_shfl<-1>(x[r + 1][E - 1]), right = fx_shfl<1>(x[r + 1][0]);
      double out[E];
      bool ok[E], all = true;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const FxV &p = x[r + 1][e], &w = e == 0 ? left : x[r + 1][e - 1],
                  &ea = e == E - 1 ? right : x[r + 1][e + 1];
        const FxV &s = x[r][e], &n = x[r + 2][e], &lo = below[r][e], &hi = up[r + 1][e];
        const int m = max(max(max(max(w.e, ea.e), max(s.e, n.e)), max(lo.e, hi.e)), p.e);
        const int64_t ns = ((fx_align(w, m) + fx_align(ea, m)) + (fx_align(s, m) + fx_align(n, m))) +
                           (fx_align(lo, m) + fx_align(hi, m));
        ok[e] = fx_update<3>(p, ns, m, coef, &out[e]);
        all = all && ok[e];
        below[r][e] = p;
      }
      if (!all) {  // some take the FP64 operations, from memory
        const double *pl = src + (int64_t)z * plane, *row = pl + ro[r + 1];
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if (ok[e]) continue;
          const int im = xi[e] > 0 ? xi[e] - 1 : 0, ip = min(xi[e] + 1, nx - 1);
          out[e] = fx_plain<3>(row[xi[e]],
                               {row[im], row[ip], pl[ro[r] + xi[e]], pl[ro[r + 2] + xi[e]],
                                src[(int64_t)max(z - 1, 0) * plane + ro[r + 1] + xi[e]], zp[ro[r + 1] + xi[e]]},
                               coef);
        }
      }
      if (y0 + r < ny) fx_store<E>(dst + (int64_t)z * plane + (int64_t)(y0 + r) * g.pitch, xl, lane, nx, out);
    }
#pragma unroll
    for (int r = 0; r < R + 2; ++r)
#pragma unroll
      for (int e = 0; e < E; ++e) x[r][e] = up[r][e];
  }
}

// Rows (planes) per item of a march.  An item converts two more rows than it
// writes and starts with a wait for memory (together `pro` rows' time), and an
// SM holds `occ` CTAs: with q CTAs to an SM a row of each takes one + add q us
// up to one full round, with more of them `full` us a round.  So for every q
// the most items that keep to it, and of these the cheapest (up to 24 CTAs to
// an SM more than the fewest: there the starts of the items outweigh the rest).
// Fitted to sweeps over chunks for 64^3 .. 256^3 and 1152^2 .. 8192^2, where the choice is
// within 4 % of the best.  One round of about 16 (2D: 24) warps an SM, rounded
// to whole items, took 24 % longer at 256^3, whose CTAs it dealt 3.2 to an SM, and
// 7 % at 8192^2.
struct FxMarch {
  int occ;
  double one, add, full, pro;
};
constexpr FxMarch kFxMarch2 = {6, 0.443, 0.314, 2.10, 0.91}, kFxMarch3 = {4, 0.705, 0.371, 2.07, 0.71};

static int64_t fx_chunk(const FxMarch &m, int64_t columns, int64_t len, int num_sms) {
  const int64_t round = (int64_t)std::max(1, num_sms) * kFxWarps;  // warps of one CTA an SM
  const int64_t q0 = (columns + round - 1) / round;
  double best[2] = {1e300, 1e300};  // one round; several
  int64_t best_chunk[2] = {len, len};
  for (int64_t qt = q0; qt < q0 + 24; ++qt) {
    const int64_t chunk = (len + qt * round / columns - 1) / (qt * round / columns);
    const int64_t warps = columns * ((len + chunk - 1) / chunk);
    const int64_t q = (warps + round - 1) / round;
    const int64_t rounds = q / m.occ, rest = q % m.occ;
    const double row = q <= m.occ ? m.one + m.add * (double)q
                                  : m.full * (double)rounds + (rest ? m.one + m.add * (double)rest : 0.0);
    const double cost = row * ((double)chunk + m.pro);
    const int several = q > m.occ;
    if (cost < best[several]) best[several] = cost, best_chunk[several] = chunk;
    if (chunk == 1) break;
  }
  return best_chunk[best[1] < 0.97 * best[0]];  // the fit's own error
}

static cudaError_t direct_fx(int ndim, const GridParams &g, const double *src, double *dst, int num_sms,
                             cudaStream_t s) {
  const int w = ndim == 2 ? kFx2W : kFx3W;
  const int64_t strips = (g.nx + w - 2 * kFxHalo - 1) / (w - 2 * kFxHalo);
  const int64_t bands = ndim == 2 ? 1 : (g.ny + kFx3R - 1) / kFx3R;
  const int64_t len = ndim == 2 ? g.ny : g.nz;
  const int64_t chunk = fx_chunk(ndim == 2 ? kFxMarch2 : kFxMarch3, strips * bands, len, num_sms);
  const int64_t warps = strips * bands * ((len + chunk - 1) / chunk);
  const unsigned blocks = (unsigned)((warps + kFxWarps - 1) / kFxWarps);
  if (ndim == 2) step2d_fx<<<blocks, kFxWarps * 32, 0, s>>>(src, dst, g, (int)strips, (int)chunk);
  else step3d_fx<<<blocks, kFxWarps * 32, 0, s>>>(src, dst, g, (int)strips, (int)bands, (int)chunk);
  return cudaGetLastError();
}

// ------------------------------------------------ small 3D FP32 grids --
// One step a launch, a thread owning a vector of 4 cells of RZ planes of one
// row: what the default 3D schedule runs on small grids.  There a pass of the
// streaming kernel takes some 11 us for its two steps whatever the size (its
// CTAs wait for one plane after another), this one little more than a launch:
// 32^3 5.4 -> 1.5 us a step, 64^3 5.5 -> 2.1, 100^3 5.5 -> 4.2 (128^3: 5.5
// against 5.9).  All loads are issued before the first use.
template <int RZ>
__global__ void __launch_bounds__(64) step3d_vec(const float *__restrict__ src, float *__restrict__ dst,
                                                 GridParams g, int nvx) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int nx = (int)g.nx, ny = (int)g.ny, nz = (int)g.nz;
  const int y = (int)(idx / nvx), x = 4 * (int)(idx - (int64_t)y * nvx);
  const int z0 = blockIdx.y * RZ;
  // The previous launch on the stream writes what this one reads.
  pdl_wait();
  if (y >= ny) return;
  const int64_t plane = g.pitch * g.ny;
  const float *p = src + z0 * plane + y * g.pitch + x;
  const int64_t ds = y > 0 ? -g.pitch : 0, dn = y + 1 < ny ? g.pitch : 0;
  const float alpha = (float)g.alpha, beta = (float)g.beta;
  float c[RZ + 2][4], s[RZ][4], n[RZ][4], l[RZ], r[RZ];
#pragma unroll
  for (int j = -1; j <= RZ; ++j) ld_cells<float, 4>(p + (min(max(z0 + j, 0), nz - 1) - z0) * plane, c[j + 1]);
#pragma unroll
  for (int j = 0; j < RZ; ++j) {
    const float *q = p + (min(z0 + j, nz - 1) - z0) * plane;
    ld_cells<float, 4>(q + ds, s[j]);
    ld_cells<float, 4>(q + dn, n[j]);
    l[j] = x > 0 ? q[-1] : c[j + 1][0];
    r[j] = x + 4 < nx ? q[4] : 0.f;
  }
  pdl_launch_dependents();
#pragma unroll
  for (int j = 0; j < RZ; ++j) {
    if (z0 + j >= nz) break;
    float out[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float m = c[j + 1][e];
      const float w = e == 0 ? l[j] : c[j + 1][e > 0 ? e - 1 : 0];
      const float ea = x + e + 1 >= nx ? m : e == 3 ? r[j] : c[j + 1][e < 3 ? e + 1 : 3];
      out[e] = ac_update<float>(m, ((w + ea) + (s[j][e] + n[j][e])) + (c[j][e] + c[j + 2][e]), -6.0f, alpha, beta);
    }
    float *q = dst + (z0 + j) * plane + y * g.pitch + x;
    if (x + 4 <= nx) {
      st_cells<float, 4>(q, out);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (x + e < nx) q[e] = out[e];
    }
  }
}

// (A streaming pass over a few large planes has short chains: 700 x 700 x 2 and
// 600 x 600 x 3 3.1 and 3.6 us a step against 3.7 and 4.4, 400 x 400 x 2 3.1 against
// 2.1.)
bool step3d_vec_serves(int dtype, const GridParams &g) {
  return dtype == AC_F32 && g.nx * g.ny * g.nz <= (g.nz < 6 ? 400000 : 1500000) && g.nz <= 65535;
}

cudaError_t launch_step3d_vec(const GridParams &g, const void *src, void *dst, cudaStream_t s) {
  const int nvx = (int)((g.nx + 3) / 4);
  // planes a thread: no more than there are
  const int64_t cells = g.nx * g.ny * g.nz;
  const int rz = cells < 64000 || g.nz < 2 ? 1 : cells < 500000 || g.nz < 4 ? 2 : 4;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((g.ny * nvx + 63) / 64), (unsigned)((g.nz + rz - 1) / rz));
  cfg.blockDim = dim3(64);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const float *a = (const float *)src;
  float *b = (float *)dst;
  switch (rz) {
    case 1: return cudaLaunchKernelEx(&cfg, step3d_vec<1>, a, b, g, nvx);
    case 2: return cudaLaunchKernelEx(&cfg, step3d_vec<2>, a, b, g, nvx);
    default: return cudaLaunchKernelEx(&cfg, step3d_vec<4>, a, b, g, nvx);
  }
}

// FP64 grids (integer form) of at most two blocks an SM are launched to overlap the previous
// launch's tail (programmatic stream serialization): 16^3 1.78 -> 1.56 us a step,
// 32^3 1.92 -> 1.76, 256^2 1.98 -> 1.85.  With more blocks the next launch's take the SMs of this one's
// (48^3 3.15 -> 3.42).
template <typename T>
static cudaError_t direct_t(int ndim, const GridParams &g, const void *src, void *dst, int num_sms,
                            cudaStream_t s) {
  const bool tall = cell_grid_tall(g);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = cell_grid(g);
  cfg.blockDim = dim3(kCellBlockX, kCellBlockY);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g.fx.limit && (int64_t)cfg.gridDim.x * cfg.gridDim.y * cfg.gridDim.z <= 2 * num_sms ? 1 : 0;
  void (*k)(const T *, T *, GridParams);
  if (ndim == 2) k = tall ? step2d_direct<T, true> : step2d_direct<T, false>;
  else k = tall ? step3d_direct<T, true> : step3d_direct<T, false>;
  return cudaLaunchKernelEx(&cfg, k, (const T *)src, (T *)dst, g);
}

cudaError_t launch_direct(int ndim, int dtype, const GridParams &g, const void *src, void *dst, int num_sms,
                          cudaStream_t s) {
  switch (dtype) {
    case AC_F64:
      if (g.fx.limit && fx_marches(ndim, g))
        return direct_fx(ndim, g, (const double *)src, (double *)dst, num_sms, s);
      return direct_t<double>(ndim, g, src, dst, num_sms, s);
    case AC_F32: return direct_t<float>(ndim, g, src, dst, num_sms, s);
    case AC_F16S: return direct_t<__half>(ndim, g, src, dst, num_sms, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ac
