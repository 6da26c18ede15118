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
// both are below 2^-5 2^E.  Otherwise the rms error, by the size of the result
// against the stencil (down to 2^-10) and for rough, smooth and planar
// stencils, is 0.03 to 0.98 of the FP64 operations', its largest value at most
// 0.95 of theirs (128-bit arithmetic, amplitudes 1e-6 .. 1.7, alpha 0.0004 ..
// 0.6, 2D and 3D).  +-1 and 0 stay exact fixed points, and mirrored or negated
// fields give the mirrored or negated result bit for bit.
// Likewise a cell whose stencil holds a value of 1.75 or more in size (fields
// of the scheme have |phi| <= 1), NaN or infinity, or none above 2^-959, and one
// that is 0, takes the FP64 operations.  The form a cell takes and its result
// depend on its stencil's values alone, so every kernel and schedule gives the
// same bits.
#pragma once

#include "common.cuh"

namespace ac {

struct Fx {  // x = hi 2^32 + lo with lo signed
  int hi, lo;
};
__device__ __forceinline__ Fx fx_split(int64_t x) {
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
__device__ __forceinline__ FxV fx_in(double v) {
  const int hi = __double2hiint(v);
  const uint32_t twice = 2u * (uint32_t)hi;  // without the sign
  const uint64_t a = ((uint64_t)(uint32_t)((hi & 0xfffff) | 0x100000) << 32 | (uint32_t)__double2loint(v)) << 9;
  FxV r;
  r.m = (int64_t)a ^ (int64_t)(hi >> 31);
  r.e = twice < 2u * 0x3ffc0000u ? (int)(twice >> 21) : kFxOut;
  return r;
}
// Whether a stencil with largest exponent e takes the integer form.
__device__ __forceinline__ bool fx_in_range(int e) { return (unsigned)(e - 64) < 1024u - 64u; }
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

// Whether alpha 2^63 and beta 2^65 fit (not for alpha near 1 or beta at the 2D
// stability limit, where every cell takes the FP64 operations).
__host__ __device__ constexpr bool fx_coefficients(double alpha, double beta) {
  return alpha < 0.99 && beta < 0.2499;
}

// Coefficients of the update for one grid; FP64: also in fixed point.
template <typename C>
struct Coef {
  C alpha, beta;
  __device__ __forceinline__ Coef(double a, double b) : alpha((C)a), beta((C)b) {}
};
template <>
struct Coef<double> {
  double alpha, beta;
  Fx A, B;
  bool fx;
  __device__ __forceinline__ Coef(double a, double b) : alpha(a), beta(b) {
    fx = fx_coefficients(a, b);
    A = fx_split(__double2ll_rn((fx ? a : 0.0) * 0x1p63));
    B = fx_split(__double2ll_rn((fx ? b : 0.0) * 0x1p65));
  }
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
  // r or 2 b of 2^55 = 2^-5 2^E units or more (high halves of 2^23)
  constexpr uint32_t kKeep = 1u << 23;
  const uint32_t big = ((uint32_t)(r >> 32) + kKeep) | (2u * (uint32_t)(b >> 32) + kKeep);
  return (big & ~(2u * kKeep - 1u)) != 0 && p.e > 0 && fx_in_range(e);
}

// The FP64 step of one cell from its neighbours, whose sum in FP64 is nsum.
// (Calls, not inlined: the streaming kernels would hold a copy per level.)
__device__ __noinline__ inline double fx_cell2(double p, double w, double e, double s, double n, double nsum,
                                               const Coef<double> &c) {
  if (c.fx) {
    const FxV x = fx_in(p), xw = fx_in(w), xe = fx_in(e), xs = fx_in(s), xn = fx_in(n);
    const int m = max(max(max(x.e, xw.e), max(xe.e, xs.e)), xn.e);
    double out;
    if (fx_update<2>(x, (fx_align(xw, m) + fx_align(xe, m)) + (fx_align(xs, m) + fx_align(xn, m)), m, c, &out)) return out;
  }
  return ac_update<double>(p, nsum, -4.0, c.alpha, c.beta);
}
__device__ __noinline__ inline double fx_cell3(double p, double w, double e, double s, double n, double b,
                                               double f, double nsum, const Coef<double> &c) {
  if (c.fx) {
    const FxV x = fx_in(p), xw = fx_in(w), xe = fx_in(e), xs = fx_in(s), xn = fx_in(n), xb = fx_in(b),
              xf = fx_in(f);
    const int m = max(max(max(x.e, xw.e), max(xe.e, xs.e)), max(xn.e, max(xb.e, xf.e)));
    double out;
    if (fx_update<3>(x, ((fx_align(xw, m) + fx_align(xe, m)) + (fx_align(xs, m) + fx_align(xn, m))) +
                             (fx_align(xb, m) + fx_align(xf, m)), m, c, &out)) return out;
  }
  return ac_update<double>(p, nsum, -6.0, c.alpha, c.beta);
}

// One explicit Euler step of a cell from its neighbours (see ac_update).
template <typename C>
__device__ __forceinline__ C cell_update2(C p, C w, C e, C s, C n, const Coef<C> &c) {
  const C nsum = (w + e) + (s + n);
  if constexpr (sizeof(C) == 8) return fx_cell2(p, w, e, s, n, nsum, c);
  else return ac_update<C>(p, nsum, C(-4), c.alpha, c.beta);
}
template <typename C>
__device__ __forceinline__ C cell_update3(C p, C w, C e, C s, C n, C b, C f, const Coef<C> &c) {
  const C nsum = ((w + e) + (s + n)) + (b + f);
  if constexpr (sizeof(C) == 8) return fx_cell3(p, w, e, s, n, b, f, nsum, c);
  else return ac_update<C>(p, nsum, C(-6), c.alpha, c.beta);
}

}  // namespace ac
