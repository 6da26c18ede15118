// FP64 updates in 64-bit integers.
//
// GB300 issues fewer than two FP64 operations per clock and SM, so the 8 (2D)
// or 10 (3D) FP64 operations of an update cap FP64 grids at 66 / 52
// Gcell-updates/s while the integer pipes idle.  The update of a cell is
// formed in block floating point instead: the values of its stencil, as
// integers in units of 2^-58 of their largest power of two 2^E (in magnitude
// cut off there and taken half a unit larger, so that the signs are alike),
//   lap      exact sums (any order gives the same bits; the halves cancel),
//   phi^2, 1 - phi^2, |phi| (1 - phi^2) and the products with alpha and beta
//            from 32 x 32 -> 64-bit multiply-adds on balanced halves,
//   phi'     = phi + beta lap + alpha (phi - phi^3), rounded once to FP64.
// The error before that rounding is about 2^-60 2^E, which the FP64
// operations (fused as in ac_update) beat where a cell much smaller than its
// neighbours stays so because theirs cancel: at a zero crossing their sums are
// exact.  There the cell takes them: when the result and its Laplacian part
// both are below 2^-5 2^E (alpha = 0: 2^-4).  Otherwise the rms error, by the size
// of the result against the stencil (down to 2^-10) and for rough, smooth and
// planar stencils, is 0.03 to 0.98 of the FP64 operations', its largest value at
// most 0.98 of theirs (128-bit arithmetic, amplitudes 1e-6 .. 1.7, alpha 0 and
// 1e-9 .. 0.6, 2D and 3D).  +-1 and 0 stay exact fixed points, and mirrored or
// negated fields give the mirrored or negated result bit for bit.
// Likewise a cell whose stencil holds a value of 1.75 or more in size (fields
// of the scheme have |phi| <= 1; in the heat equation, alpha = 0: 2^340), NaN or
// infinity, or none above 2^-959, and one that is 0, takes the FP64 operations.
// (A field that is all beyond 1.75 is formed twice: 4096^2 348 us a step against
// 253 by the FP64 operations alone.  A test that spares it the first form cost
// every field 2.5 %.)
// The form a cell takes and its result depend on its stencil's values alone, so
// every kernel and schedule gives the same bits.
#pragma once

#include <cmath>

#include "common.cuh"

namespace ac {

struct Fx {  // x = hi 2^32 + lo with lo signed
  int hi, lo;
};
__host__ __device__ __forceinline__ Fx fx_split(int64_t x) {
  Fx r;
  r.lo = (int)(uint32_t)x;
  r.hi = (int)(x >> 32) + (int)((uint32_t)x >> 31);
  return r;
}
// a * b / 2^64, rounded; the product of the low halves (a quarter of a unit
// at most) is left out.  Three wide multiply-adds and a sign extension, in
// PTX: from C the same arithmetic took 13 instructions.
__device__ __forceinline__ int64_t fx_mulhi(const Fx &a, const Fx &b) {
  int64_t r;
  asm("{\n\t.reg .s64 t, u;\n\t.reg .s32 l, h;\n\t"
      "mad.wide.s32 t, %1, %4, %5;\n\t"
      "mad.wide.s32 t, %2, %3, t;\n\t"
      "mov.b64 {l, h}, t;\n\t"
      "cvt.s64.s32 u, h;\n\t"
      "mad.wide.s32 %0, %1, %3, u;\n\t}"
      : "=l"(r)
      : "r"(a.hi), "r"(a.lo), "r"(b.hi), "r"(b.lo), "l"(0x80000000ll));
  return r;
}

// A value as m 2^(e - 1084), 2^61 <= m < 2^62, or ~m for a negative one, so
// that shifts to the right cut both off alike (0 and subnormal values: any m,
// e = 0); e = kFxOut for one that is out of range.
struct FxV {
  int64_t m;
  int e;
};
constexpr int kFxOut = 2047;
// (Integer instructions only: the conversions from and to 64-bit integers
// are slower than the FP64 operations they would replace.)
__device__ __forceinline__ FxV fx_in(double v, uint32_t limit) {
  const int hi = __double2hiint(v);
  const uint32_t twice = 2u * (uint32_t)hi;  // without the sign
  const uint64_t a = ((uint64_t)(uint32_t)((hi & 0xfffff) | 0x100000) << 32 | (uint32_t)__double2loint(v)) << 9;
  FxV r;
  r.m = (int64_t)a ^ (int64_t)(hi >> 31);
  r.e = twice < limit ? (int)(twice >> 21) : kFxOut;
  return r;
}
// Whether a stencil with largest exponent e takes the integer form.
__device__ __forceinline__ bool fx_in_range(int e) { return (unsigned)(e - 64) < (unsigned)(kFxOut - 64); }
// m / 2^d, d >= 0, rounded down (the instruction clamps d).
__device__ __forceinline__ int64_t fx_shift(int64_t m, int d) {
  int64_t r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(d));
  return r;
}
// v in units of 2^(e - 1081), e at least its exponent: y for y + 1/2.
__device__ __forceinline__ int64_t fx_align(const FxV &v, int e) { return fx_shift(v.m, e - v.e + 3); }
// (negative ? -1 : 1) x 2^(e - 1083), rounded once: x's halves become the
// mantissas of doubles with those units and 2^32 times them, less the constant
// that their leading bits (and the high half's offset 2^31) stand for; the
// first sum is exact.
__device__ __forceinline__ double fx_out(int64_t x, int e, int negative) {
  const double lo = __hiloint2double((e - 8) << 20, (int)(uint32_t)x);
  const double hi = __hiloint2double((e + 24) << 20, (int)((uint32_t)(x >> 32) ^ 0x80000000u));
  const double r = __dadd_rn(__dsub_rn(hi, __hiloint2double((e + 24) << 20, (int)0x80100000u)), lo);
  return __hiloint2double(__double2hiint(r) ^ (negative & (int)0x80000000u), __double2loint(r));
}

template <int D>
__device__ __forceinline__ FxV fx_shfl(const FxV &v) {  // of the lane D above
  FxV r;
  r.m = D > 0 ? __shfl_down_sync(0xffffffffu, v.m, D) : __shfl_up_sync(0xffffffffu, v.m, -D);
  r.e = D > 0 ? __shfl_down_sync(0xffffffffu, v.e, D) : __shfl_up_sync(0xffffffffu, v.e, -D);
  return r;
}

// The fixed-point coefficients of a grid (formed on the host: the conversions
// take longer than an update).
inline FxCoef fx_coef(double alpha, double beta) {
  FxCoef c{};
  if (!(alpha < 0.99 && beta < 0.2499)) return c;
  const Fx a = fx_split((int64_t)std::llrint(alpha * 0x1p63)), b = fx_split((int64_t)std::llrint(beta * 0x1p65));
  c.ah = a.hi;
  c.al = a.lo;
  c.bh = b.hi;
  c.bl = b.lo;
  // 2^55 units, 2^-5 2^E; twice that where the FP64 operations round once less
  c.keep = alpha > 0.0 ? 1u << 23 : 1u << 24;
  // 1.75: phi (1 - phi^2) stays below 4; 2^340: phi^3 stays finite
  c.limit = 2u * (alpha > 0.0 ? 0x3ffc0000u : 1363u << 20);
  return c;
}

// Coefficients of the update for one grid, from its GridParams or BInst; FP64:
// also in fixed point.
template <typename C>
struct Coef {
  C alpha, beta;
  template <typename P>
  __device__ __forceinline__ explicit Coef(const P &g) : alpha((C)g.alpha), beta((C)g.beta) {}
};
template <>
struct Coef<double> {
  double alpha, beta;
  Fx A, B;
  uint32_t limit, keep;
  template <typename P>
  __device__ __forceinline__ explicit Coef(const P &g)
      : alpha(g.alpha), beta(g.beta), A{g.fx.ah, g.fx.al}, B{g.fx.bh, g.fx.bl}, limit(g.fx.limit), keep(g.fx.keep) {}
};

// The updated cell from p, the sum of its neighbours' fx_align and the
// stencil's largest exponent e, in *out; whether that is the cell's result
// (false: it takes the FP64 operations).  Formed for |p|, with the Laplacian's
// sign turned along, and the sign put back.
template <int NDIM>
__device__ __forceinline__ bool fx_update(const FxV &p, int64_t nsum, int e, const Coef<double> &c, double *out) {
  const int neg = (int)(p.m >> 32) >> 31;
  const int64_t s = neg, y = fx_align(p, e), x = y ^ s;
  const int64_t lap = ((nsum - (NDIM == 2 ? y << 2 : (y << 2) + (y << 1))) ^ s) - s;
  const Fx P = fx_split(p.m ^ s);
  // 1 - phi^2 in units of 2^-58, |phi| times it in 2^(p.e - 1078)
  const int64_t w = (1ll << 58) - fx_shift(fx_mulhi(P, P), 2046 - 2 * p.e);
  const int64_t q = fx_mulhi(P, fx_split(w));
  const int64_t a = fx_mulhi(fx_split(q << 6), c.A);  // units 2^(p.e - 1083)
  const int64_t b = fx_mulhi(fx_split(lap), c.B);     // units 2^(e - 1082)
  const int64_t r = (x << 2) + (b << 1) + fx_shift(a, e - p.e);
  *out = fx_out(r, e, neg);
  // r or 2 b large enough, their high halves c.keep (a power of two) or more
  const uint32_t big = ((uint32_t)(r >> 32) + c.keep) | (2u * (uint32_t)(b >> 32) + c.keep);
  return big >= 2u * c.keep && p.e > 0 && fx_in_range(e);
}

// The FP64 operations of a cell (see ac_update) from its neighbours w, e, s, n
// [, b, f].  Beside the integer form, zeros all round give 0 without them: whole
// regions of a field may be at rest (4096^2 of zeros 348 us a step with them, 137
// without).
template <int NDIM>
__device__ __forceinline__ double fx_plain(double p, const double (&v)[2 * NDIM], const Coef<double> &c) {
  if (c.limit) {
    int64_t any = __double_as_longlong(p);
#pragma unroll
    for (int d = 0; d < 2 * NDIM; ++d) any |= __double_as_longlong(v[d]);
    if (any << 1 == 0) return 0.0;
  }
  double nsum = (v[0] + v[1]) + (v[2] + v[3]);
  if constexpr (NDIM == 3) nsum = nsum + (v[4] + v[5]);
  return ac_update<double>(p, nsum, -2.0 * NDIM, c.alpha, c.beta);
}

// One explicit Euler step of a cell from its neighbours.
template <int NDIM>
__device__ __forceinline__ double fx_cell(double p, const double (&v)[2 * NDIM], const Coef<double> &c) {
  if (c.limit) {
    const FxV x = fx_in(p, c.limit);
    FxV f[2 * NDIM];
    int m = x.e;
#pragma unroll
    for (int d = 0; d < 2 * NDIM; ++d) {
      f[d] = fx_in(v[d], c.limit);
      m = max(m, f[d].e);
    }
    int64_t ns = 0;
#pragma unroll
    for (int d = 0; d < 2 * NDIM; ++d) ns += fx_align(f[d], m);
    double out;
    if (fx_update<NDIM>(x, ns, m, c, &out)) return out;
  }
  return fx_plain<NDIM>(p, v, c);
}

// The same of a lane's E adjacent cells: row[0] and row[E + 1] are the cells
// beside them, y[d] the other neighbours s, n [, b, f].  Only cells x0 + e in
// [0, nx) are read by anyone: the zeros that lie outside the grid don't send the
// warp through the FP64 operations.
template <int NDIM, int E>
struct FxCells {
  double row[E + 2], y[2 * NDIM - 2][E];
};
template <int E>
struct FxResult {
  double v[E];
};
template <int NDIM, int E>
__device__ __forceinline__ FxResult<E> fx_cells(const FxCells<NDIM, E> &in, const Coef<double> &c, int x0, int nx) {
  FxResult<E> out;
  bool ok[E], all = false;
  if (c.limit) {
    all = true;
    FxV x[E + 2];
#pragma unroll
    for (int e = 0; e < E + 2; ++e) x[e] = fx_in(in.row[e], c.limit);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      FxV f[2 * NDIM - 2];
      int m = max(max(x[e].e, x[e + 1].e), x[e + 2].e);
#pragma unroll
      for (int d = 0; d < 2 * NDIM - 2; ++d) {
        f[d] = fx_in(in.y[d][e], c.limit);
        m = max(m, f[d].e);
      }
      int64_t ns = fx_align(x[e], m) + fx_align(x[e + 2], m);
#pragma unroll
      for (int d = 0; d < 2 * NDIM - 2; ++d) ns += fx_align(f[d], m);
      ok[e] = fx_update<NDIM>(x[e + 1], ns, m, c, &out.v[e]);
      all = all && ok[e];
    }
  }
  if (!all) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if ((c.limit && ok[e]) || (unsigned)(x0 + e) >= (unsigned)nx) continue;
      double v[2 * NDIM] = {in.row[e], in.row[e + 2]};
#pragma unroll
      for (int d = 0; d < 2 * NDIM - 2; ++d) v[d + 2] = in.y[d][e];
      out.v[e] = fx_plain<NDIM>(in.row[e + 1], v, c);
    }
  }
  return out;
}

// As a call: the 2D streaming kernels would hold a copy per level and unrolled
// row, and run out of instruction cache.
template <int NDIM, int E>
__device__ __noinline__ FxResult<E> fx_cells_call(FxCells<NDIM, E> in, Coef<double> c, int x0, int nx) {
  return fx_cells<NDIM, E>(in, c, x0, nx);
}

}  // namespace ac
