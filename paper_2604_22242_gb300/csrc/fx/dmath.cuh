// dmath.cuh - FP64 exp, sqrt and division that spend few FP64 instructions.
//
// This part issues one warp-wide FP64 instruction per SM sub-partition in
// about 64 cycles, 64 times the FP32 and integer cost, so an FP64 tree with
// transcendentals is bound by how many FP64 instructions an element needs
// and by nothing else. Here the seeds, reductions and small terms run in FP32
// and integer arithmetic, and FP64 is kept for the steps that carry the full
// precision:
//
//   exp   4 FP64 instructions. Table-driven (P. T. P. Tang, "Table-driven
//         implementation of the exponential function in IEEE floating-point
//         arithmetic", ACM TOMS 15(2), 1989) with 1024 entries:
//         x = n ln2/1024 + r, |r| < 4.3e-4, exp(x) = 2^(n/1024) (1 + p),
//         p = r (1 + r/2) + small, where small = r^3/6 + r^4/24 - n c2 + lo
//         (c2 the part of ln2/1024 below FP64, lo the table entry's
//         remainder) is below 1e-10 and so needs only FP32.
//   sqrt  3 FP64 instructions. FP32 square root with an FP32 correction (a
//         pair good to about 2^-45), then one Newton step with the exact
//         FP64 residual.
//   div   3 FP64 instructions, the same way from the FP32 reciprocal.
//
// X % Y + sqrt(abs(W)) / (1 + exp(-V)) needs 12 FP64 instructions an element
// this way and 35 with CUDA's functions: 0.28 ms at 3001 x 4096, where FP64
// sign changes (expr.cuh) took it to 14 and 0.34 ms.
//
// The last step of sqrt and div adds a correction of relative size 2^-45 that
// is known to a relative error of 2^-21. Where the sum comes within 2^-11 ulp of
// a tie between two results (one argument in 1024; near_tie, a dozen FP32 and
// integer instructions) the exact residual of the result decides, one FP64
// instruction more, so both are correctly rounded, as CUDA's are. exp is within
// 0.6 ulp. (With the CUDA functions called in these cases instead, which take ten
// FP64 instructions and more, Z of the statistics at 3001 x 4096 took 284 us
// against 275; without any of it, 272.)
// Arguments outside the ranges named at each function (infinities, NaN,
// zeros, subnormals, extreme exponents) take the CUDA function or operator,
// out of line. Reference tests run these functions on the host against
// extended precision (the host seeds are an FP32 division and square root,
// perturbed).
#pragma once

#include <cstdint>
#include <cstring>

#include "core.cuh"

namespace fx {
namespace dm {

struct alignas(16) Exp2Row {
  double t;
  float lo;
  int pad;
};
static __device__ const Exp2Row kExp2Rows[1024] = {
#include "exp2_table.inc"
};

// ---------------------------------------------------------------- bits

FX_HD uint32_t hi_word(double x) {
#ifdef __CUDA_ARCH__
  return uint32_t(__double2hiint(x));
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return uint32_t(b >> 32);
#endif
}
FX_HD uint32_t lo_word(double x) {
#ifdef __CUDA_ARCH__
  return uint32_t(__double2loint(x));
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return uint32_t(b);
#endif
}
FX_HD double from_words(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(int(hi), int(lo));
#else
  const uint64_t b = (uint64_t(hi) << 32) | lo;
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
FX_HD float f32_of(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  memcpy(&x, &b, 4);
  return x;
#endif
}
FX_HD uint32_t bits_of(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  memcpy(&b, &x, 4);
  return b;
#endif
}

FX_HD float ffma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return __builtin_fmaf(a, b, c);
#endif
}
FX_HD double dfma(double a, double b, double c) {
#ifdef __CUDA_ARCH__
  return __fma_rn(a, b, c);
#else
  return __builtin_fma(a, b, c);
#endif
}
FX_HD double dadd(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dadd_rn(a, b);
#else
  return a + b;
#endif
}
// FP32 seeds: the hardware's approximations (about 2^-23 relative). On the
// host, a division or square root moved by two ulps stands in for them.
FX_HD float seed_rcp(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return f32_of(bits_of(1.0f / x) + 2u);
#endif
}
FX_HD float seed_rsqrt(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return f32_of(bits_of(1.0f / __builtin_sqrtf(x)) - 2u);
#endif
}
FX_HD Exp2Row exp2_row(uint32_t j) {
#ifdef __CUDA_ARCH__
  const int4 q = __ldg(reinterpret_cast<const int4*>(kExp2Rows) + j);
  return Exp2Row{__hiloint2double(q.y, q.x), __int_as_float(q.z), 0};
#else
  static const Exp2Row rows[1024] = {
#include "exp2_table.inc"
  };
  return rows[j];
#endif
}

// x cut to FP32 precision (toward zero); x must be below 2^127 in magnitude,
// and below 2^-95 counts as zero. Integer instructions only: the conversion
// instruction runs at the FP64 rate.
FX_HD float cut(double x) {
  const uint32_t h = hi_word(x), l = lo_word(x);
  const uint32_t b = ((h - 0x38000000u) << 3) | (l >> 29);
  const float f = f32_of((b & 0x7FFFFFFFu) | (h & 0x80000000u));
  return (h & 0x7FFFFFFFu) < 0x3A000000u ? 0.0f : f;
}
// A normal FP32 value as FP64; zero becomes 2^-127 (of f's sign).
FX_HD double widen_bits(float f) {
  const uint32_t b = bits_of(f);
  return from_words((((b & 0x7FFFFFFFu) >> 3) + 0x38000000u) | (b & 0x80000000u), b << 29);
}

// May s, the rounded sum of Q and a correction t, not be the nearest one? (t to
// FP32 precision, Q within 2^9 steps of s, both positive and of magnitude near 1;
// ulps the steps of s in a unit.) True when the sum may be nearer than 2^-11 of a
// step to the middle between two results.
FX_HD bool near_tie(double s, double Q, float t, float ulps) {
  const float k = f32_of(0x4B400000u + (lo_word(s) - lo_word(Q))) - 12582912.0f;  // steps from Q to s
  return f32_of(bits_of(ffma(t, ulps, -k)) & 0x7FFFFFFFu) >= 0.5f - 0x1p-11f;
}
// The steps from Q to s are all of one length: one exponent, and not a power
// of two, below which they are half as long.
FX_HD bool one_binade(double s, double Q) {
  return (hi_word(s) ^ hi_word(Q)) < 0x00100000u && ((hi_word(s) & 0x000FFFFFu) | lo_word(s)) != 0u;
}
FX_HD uint64_t bits64(double x) { return (uint64_t(hi_word(x)) << 32) | lo_word(x); }
FX_HD double step_to(double s, bool up) {
  const uint64_t b = bits64(s) + (up ? 1u : ~uint64_t(0));
  return from_words(uint32_t(b >> 32), uint32_t(b));
}

#ifdef __CUDACC__
static __device__ __noinline__ double exp_any(double x) { return ::exp(x); }
static __device__ __noinline__ double sqrt_any(double x) { return ::sqrt(x); }
static __device__ __noinline__ double div_any(double a, double b) { return a / b; }
#endif

// ---------------------------------------------------------------- exp

// |x| < 700 (never NaN or infinite): no overflow or subnormal result.
FX_HD bool exp_fast_ok(double x) { return (hi_word(x) & 0x7FFFFFFFu) < 0x4085E000u; }
FX_HD double exp_fast(double x) {
  const float t = ffma(cut(x), 0x1.715476p+10f, 12582912.0f);  // n = round(x 1024 / ln 2)
  const int n = int(bits_of(t) - 0x4B400000u);
  const float nf = t - 12582912.0f;
  const Exp2Row row = exp2_row(uint32_t(n) & 1023u);
  const double r = dfma(widen_bits(nf), -0x1.62e42fefa39efp-11, x);
  const float rf = cut(r);
  const float r2 = rf * rf;
  const float q = ffma(rf, 0x1.555556p-5f, 0x1.555556p-3f);  // 1/6 + r/24
  const float small = ffma(r2 * rf, q, ffma(nf, -0x1.abc9e4p-66f, row.lo));
  const double u = dfma(0.5, r, 1.0);
  const double p = dfma(r, u, widen_bits(small));
  const double s = from_words(hi_word(row.t) + (uint32_t(n >> 10) << 20), lo_word(row.t));
  return dfma(s, p, s);
}

// ---------------------------------------------------------------- sqrt

// Positive, normal and finite.
FX_HD bool sqrt_fast_ok(double x) { return hi_word(x) - 0x00100000u < 0x7FE00000u; }
FX_HD double sqrt_fast(double x, bool& sure) {
  const uint32_t h = hi_word(x), l = lo_word(x);
  const uint32_t e = ((h >> 20) - 1023u) & ~1u;  // even exponent (two's complement)
  const double m = from_words(h - (e << 20), l);  // x = m 2^e, m in [1, 4)
  const float mf = f32_of(((hi_word(m) - 0x38000000u) << 3) | (l >> 29));
  const float ml = float(l & 0x1FFFFFFFu) * (hi_word(m) >= 0x40000000u ? 0x1p-51f : 0x1p-52f);
  const float y = seed_rsqrt(mf);
  const float g = mf * y, hy = 0.5f * y;
  const float gl = (ffma(-g, g, mf) + ml) * hy;
  const double G = dadd(widen_bits(g), widen_bits(gl));
  const double d = dfma(-G, G, m);
  double s = dfma(d, widen_bits(hy), G);
  sure = one_binade(s, G) || bits64(s) == 0x3FF0000000000000u;  // exact at 1: below it there is no root
  if (near_tie(s, G, cut(d) * hy, 0x1p52f)) {
    // with u = 2^-52, m > (s + u/2)^2 = s^2 + s u + u^2/4 exactly when the residual
    // m - s^2, a multiple of u^2, is above s u; below (s - u/2)^2 when at most -s u
    const double r = dfma(-s, s, m), su = from_words(hi_word(s) - (52u << 20), lo_word(s));
    const bool up = (hi_word(r) & 0x80000000u) == 0u;
    const uint64_t rb = bits64(r) & ~(uint64_t(1) << 63);
    if (up ? rb > bits64(su) : rb >= bits64(su)) s = step_to(s, up);
  }
  return from_words(hi_word(s) + ((e << 19) & 0xFFF00000u), lo_word(s));
}

FX_HD double sqrt_fast(double x) {
  bool sure;
  return sqrt_fast(x, sure);
}

// ---------------------------------------------------------------- division

// Both magnitudes in [2^-400, 2^400): neither the quotient nor a residual
// leaves the normal range.
FX_HD bool div_fast_ok(double a, double b) {
  constexpr uint32_t lo = (1023u - 400u) << 20, span = 800u << 20;
  return (hi_word(a) & 0x7FFFFFFFu) - lo < span && (hi_word(b) & 0x7FFFFFFFu) - lo < span;
}
FX_HD double div_fast(double a, double b, bool& sure) {
  const uint32_t ha = hi_word(a), la = lo_word(a), hb = hi_word(b), lb = lo_word(b);
  // magnitudes in [1, 2); the sign and the exponents go back on at the end
  const uint32_t ma = (ha & 0x000FFFFFu) | 0x3FF00000u, mb = (hb & 0x000FFFFFu) | 0x3FF00000u;
  const double A = from_words(ma, la), B = from_words(mb, lb);
  const float af = f32_of(((ma - 0x38000000u) << 3) | (la >> 29));
  const float bf = f32_of(((mb - 0x38000000u) << 3) | (lb >> 29));
  const float al = float(la & 0x1FFFFFFFu) * 0x1p-52f, bl = float(lb & 0x1FFFFFFFu) * 0x1p-52f;
  const float y = seed_rcp(bf);
  const float q = af * y;
  const float ql = (ffma(-q, bf, af) + ffma(-q, bl, al)) * y;
  const double Q = dadd(widen_bits(q), widen_bits(ql));
  const double R = dfma(-Q, B, A);
  double s = dfma(R, widen_bits(y), Q);
  const bool ge1 = hi_word(s) >= 0x3FF00000u;
  sure = one_binade(s, Q) || (bits64(R) << 1) == 0u;
  if (near_tie(s, Q, cut(R) * y, ge1 ? 0x1p52f : 0x1p53f)) {
    // the nearest one unless A - s B exceeds half a step times B (never equal:
    // no quotient lies midway)
    const double r = dfma(-s, B, A), half = from_words(hi_word(B) - ((ge1 ? 53u : 54u) << 20), lo_word(B));
    if ((bits64(r) & ~(uint64_t(1) << 63)) > bits64(half)) s = step_to(s, (hi_word(r) & 0x80000000u) == 0u);
  }
  const uint32_t e = (ha & 0x7FF00000u) - (hb & 0x7FF00000u);
  return from_words((hi_word(s) + e) ^ ((ha ^ hb) & 0x80000000u), lo_word(s));
}

FX_HD double div_fast(double a, double b) {
  bool sure;
  return div_fast(a, b, sure);
}

}  // namespace dm
}  // namespace fx
