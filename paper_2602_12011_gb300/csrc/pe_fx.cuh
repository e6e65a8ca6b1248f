// pe_fx.cuh -- fixed-point arithmetic of the FP64 path's response geometry.
//
// Why: GB300's FP64 pipe retires 1.67 operations per SM and clock (measured loops, FMA, MUL and ADD
// alike), its FP32 pipe 122, and its integer pipes about 16 32x32->64-bit multiply-adds (IMAD.WIDE) and
// about 80 additions or shifts. The response's quantities (sines and cosines, unit-vector
// projections, sincs, third-spacecraft phases) are bounded by a few units, so a 64-bit fixed-point
// number holds them to 2^-60, finer than FP64's 2^-53, and a product of two costs three IMAD.WIDE
// (5.1 per SM and clock measured, three times an FP64 operation's rate), a sum of products three per term, an
// addition two integer adds. What is left on the FP64 pipe is what needs its range: the TaylorF2
// phase, t_f, the amplitudes and the weighted sums.
//
// Formats: fx is a signed 64-bit integer in units of 2^-60 (Q60: |value| < 8); a turn count modulo
// one turn is an unsigned 64-bit integer in units of 2^-64 turn, which wraps by itself.
#pragma once
#include "pe_df.cuh"

namespace pe {

using fx = long long;
using fxu = unsigned long long;
constexpr fx kFxOne = 1LL << 60;

// 32 x 32 -> 64-bit products. Stated in PTX: from C++ the compiler loses the operands' widths (a masked or shifted
// 64-bit value) and issues 64 x 64-bit multiplications, two to three times the instructions.
__device__ __forceinline__ fx fx_mulw(int a, int b) {
  fx r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ fx fx_madw(int a, int b, fx c) {
  fx r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// A Q60 number of magnitude below 2 split for multiplication: x = h 2^30 + l, 0 <= l < 2^30.
struct fxs {
  int h, l;
};
__device__ __forceinline__ fxs fx_split(fx x) { return fxs{(int)(x >> 30), (int)(x & 0x3fffffff)}; }

// Running sum of products: value = h + c 2^-30 (in 2^-60). The l x l products (below 2^-60) are
// dropped. c holds sums of |a| + |b| <= 8 over the terms (each term adds at most (|a| + |b|) 2^60).
// c starts at kFxHalf plus N kFxLL, the last shift's rounding and the N dropped products' means (a quarter unit
// each): rounded down instead, errors of one sign added up over a grid's bins (64-bit reference, 24 samples: a
// gradient's t_c component 3.5e-12 off, now 7.7e-13, FP64 8.0e-13).
struct fxa {
  fx h, c;
};
constexpr int kFxHalf = 1 << 29, kFxLL = 1 << 28;
template <int N = 1>   // N: the terms of the sum that this product begins
__device__ __forceinline__ fxa fx_prod(fxs a, fxs b) {
  return fxa{fx_mulw(a.h, b.h), fx_madw(a.h, b.l, fx_madw(a.l, b.h, kFxHalf + N * kFxLL - 1))};   // - 1: two products of zeros sum to 0
}
__device__ __forceinline__ void fx_mac(fxa& s, fxs a, fxs b) {
  s.h = fx_madw(a.h, b.h, s.h);
  s.c = fx_madw(a.l, b.h, fx_madw(a.h, b.l, s.c));
}
__device__ __forceinline__ fx fx_val(fxa s) { return s.h + (s.c >> 30); }
__device__ __forceinline__ fx fx_mul(fxs a, fxs b) { return fx_val(fx_prod(a, b)); }
// a b - c d (the dropped products' means cancel); M: quarter units added
template <int M = 0>
__device__ __forceinline__ fx fx_msub(fxs a, fxs b, fxs c, fxs d) {
  const fxa s = fx_prod<M>(a, b);
  return (s.h - fx_mulw(c.h, d.h)) + ((s.c - fx_madw(c.h, d.l, fx_mulw(c.l, d.h))) >> 30);
}
// Sums of N squares: the two cross products are equal, and c counts one (the dropped squares' mean is a third)
template <int N>
__device__ __forceinline__ fxa fx_sq0() {
  return fxa{0, kFxLL + N * (fx)(kFxHalf / 3)};
}
__device__ __forceinline__ void fx_macsq(fxa& s, fxs a) {
  s.h = fx_madw(a.h, a.h, s.h);
  s.c = fx_madw(a.h, a.l, s.c);
}
__device__ __forceinline__ fx fx_valsq(fxa s) { return s.h + (s.c >> 29); }

// v 2^sh as an integer (truncated towards zero) for a double v, from its bits: no FP64 operation.
// |v| 2^sh < 2^63.
__device__ __forceinline__ fx fx_from_bits(double v, int sh) {
  const fxu u = (fxu)__double_as_longlong(v);
  const fxu m = (u & 0xfffffffffffffULL) | 0x10000000000000ULL;
  const int s = (int)((u >> 52) & 0x7ff) - 1075 + sh;
  fx r = s >= 0 ? (fx)(m << (s & 63)) : (fx)(m >> (s < -63 ? 63 : -s));
  return (fx)u < 0 ? -r : r;
}
// v turns modulo one turn (|v| < 2^52)
__device__ __forceinline__ fxu fx_turns(double v) { return (fxu)fx_from_bits(v, 64); }

// f t modulo one turn for f > 0: the 106-bit product of the significands, shifted to units of 2^-64 turn (the exact
// product's bits below that are dropped; |f t| < 2^62, below 2^-63 it counts as 0).
__device__ __forceinline__ fxu fx_cycles(double f, double t) {
  const fxu uf = (fxu)__double_as_longlong(f), ut = (fxu)__double_as_longlong(t);
  const fxu mf = (uf << 11) | 0x8000000000000000ULL, mt = (ut << 11) | 0x8000000000000000ULL;
  const fxu hi = __umul64hi(mf, mt), lo = mf * mt;              // f t = (hi 2^64 + lo) 2^(ef + et - 126)
  const int s = 62 + 2 * 1023 - (int)(uf >> 52) - (int)((ut >> 52) & 0x7ff);
  fxu r = s >= 64 ? hi >> min(s - 64, 63) : (lo >> (s & 63)) | ((hi << 1) << (63 - (s & 63)));
  if (s > 126) r = 0;
  return (fx)ut < 0 ? 0 - r : r;
}

// A double word of magnitude below 2^-8 and low word below 2^-30 (1.5 2^-30 in sum with the remainder's 2^-31, so
// that the integers' sum holds) as Q60: its high word's multiple of 2^-30 by the rounding
// constant, the rest (below 2^-30) converted to an integer.
__device__ __forceinline__ fx fx_from_dw(df x) {
  const float kM = 0.01171875f;   // 1.5 2^-7: one unit in the last place is 2^-30
  const float k = __fadd_rn(x.x, kM);
  const int n = __float_as_int(k) - __float_as_int(kM);
  const float r = __fsub_rn(x.x, __fsub_rn(k, kM));   // exact
  constexpr float k60 = 1.152921504606846976e18f;
  return ((fx)n << 30) + (fx)(__float2int_rn(__fmul_rn(r, k60)) + __float2int_rn(__fmul_rn(x.y, k60)));
}

// Entries of the tables built once per detector (k_fx_tables).
struct alignas(16) FxCis {       // the angle 2 pi j / kSinTab: cos and sin in Q60, and both as double words
  fx c, s;
  float4 w;          // cos hi, cos lo, sin hi, sin lo
};
struct alignas(32) FxSinc {      // sinc about u_j = j / kFxSincPerUnit: value in Q60, derivatives f^(k)(u_j)/k!
  fx s0;
  float2 s1, s2;     // double words
  float s3, s4;
};
constexpr int kFxSincBits = 9;                                  // 512 entries per unit of u
constexpr int kFxSincPerUnit = 1 << kFxSincBits;
constexpr int kFxSincMax = 8;                                   // u < 8 (a = pi f L < 4)
constexpr int kFxSincTab = kFxSincPerUnit * kFxSincMax + 2;

// (cos, sin) of 2 pi u 2^-64: the nearest of kSinTab tabulated angles and the remainder t,
// |t| <= pi/kSinTab, by the angle-addition formulas. The table's values are Q60; what is added to
// them is below 2^-8, so double words (2^-47 relative) keep the sum to 2^-55, on the FP32 pipe.
// Not inlined, as fx_sinc: one copy each keeps the unit's loop in the instruction cache.
struct fxc {
  fx c, s;
};
static __device__ __noinline__ fxc fx_cis(fxu u, const FxCis* __restrict__ tab) {
  const fxu jr = u + (1ULL << 53);
  const fx d = (fx)(u - (jr & 0xffc0000000000000ULL));          // signed remainder, |d| <= 2^53
  const FxCis e = tab[jr >> 54];
  // d 2^-64 turns as a double word (24 bits of 2^-34, then the rest), times 2 pi
  const df dw = df_make(__fmul_rn(__int2float_rn((int)(d >> 30)), 5.8207660913467407e-11f),
                        __fmul_rn(__int2float_rn((int)d & 0x3fffffff), 5.4210108624275222e-20f));
  const df t = dfl_mul(dw, df_make(6.28318548202514648f, -1.74845553e-07f));
  const df t2 = dfl_mul(t, t);
  // cos t - 1 = t^2 (-1/2 + t^2/24) and sin t - t = t^3 (-1/6 + t^2/120) (dropped terms below 2e-18)
  const df ce = dfl_mul(t2, df_make(-0.5f, __fmul_rn(t2.x, 1.0f / 24.0f)));
  const df st = dfl_add_o(t, dfl_mul(t, dfl_mul(t2, df_make(-0.166666672f, __fmaf_rn(t2.x, 1.0f / 120.0f, 4.96705388e-09f)))));
  const df cj = df_make(e.w.x, e.w.y), sj = df_make(e.w.z, e.w.w);
  return fxc{e.c + fx_from_dw(dfl_sub(dfl_mul(cj, ce), dfl_mul(sj, st))),
             e.s + fx_from_dw(dfl_add(dfl_mul(sj, ce), dfl_mul(cj, st)))};
}

// sinc(u) = sin u / u for u = 4 u4, 0 <= u < kFxSincMax (a value below 0 by rounding counts as 0): Taylor
// series about the nearest table point, |u - u_j| <= 2^-10, through the fourth order (the fifth is
// below 2^-59). The correction to the table's value is below 2^-11 and is formed in double words;
// from the second order on the next coefficients enter the low word.
__device__ __forceinline__ fx fx_sinc(fx u4, const FxSinc* __restrict__ tab) {
  constexpr int kS = 58 - kFxSincBits;
  const int j = min(max((int)((u4 + (1LL << (kS - 1))) >> kS), 0), kFxSincTab - 1);
  const fx d = u4 - ((fx)j << kS);                               // in 2^-58 of u
  const FxSinc e = tab[j];
  const df x = df_make(__fmul_rn(__int2float_rn((int)(d >> 25)), 1.16415321826934814e-10f),          // 2^-33
                       __fmul_rn(__int2float_rn((int)d & 0x1ffffff), 3.4694469519536142e-18f));      // 2^-58
  const df p = dfl_add(e.s1, dfl_mul(x, df_make(e.s2.x, __fmaf_rn(x.x, __fmaf_rn(x.x, e.s4, e.s3), e.s2.y))));
  return e.s0 + fx_from_dw(dfl_mul(x, p));
}
// sinc of two arguments at once: each is a chain of dependent double-word operations, and two fill each other's gaps
struct fx2 {
  fx p, m;
};
static __device__ __noinline__ fx2 fx_sinc2(fx p, fx m, const FxSinc* __restrict__ tab) {
  return fx2{fx_sinc(p, tab), fx_sinc(m, tab)};
}

// 1/sqrt(x) for Q60 x in [1/2, 2): a float seed y (24 bits, taken to 2^-30), then y + y (e/2 + 3 e^2/8)
// with e = 1 - x y^2 (|e| < 2^-20; the dropped e^3 term is below 2^-61).
__device__ __forceinline__ fx fx_rsqrt(fx x) {
  const fxs xs = fx_split(x);
  const int Y = __float2int_rn(__fmul_rn(rsqrtf(__fmul_rn(__int2float_rn(xs.h), 9.3132257461547852e-10f)), 1073741824.0f));
  const fxs y2 = fx_split(fx_mulw(Y, Y));
  const fx e = kFxOne - fx_mul(xs, y2);                          // below 2^40 in magnitude
  const int t = (int)((e + (1 << 25)) >> 26);                                  // e in 2^-34: 14 bits
  const fx q = ((e << 10) + 3 * t * t + 1024) >> 11;             // e/2 + 3 e^2/8 (to 2^-58)
  const fxs qs = fx_split(q);
  return fx_madw(Y, qs.h, (fx)Y << 30) + (fx_madw(Y, qs.l, kFxHalf) >> 30);
}

}  // namespace pe
