// FP64-accurate arithmetic on the integer pipes.
//
// On GB300 a warp's FP64 instruction holds its sub-partition's FP64 unit for
// 64 cycles, a 32 x 32 -> 64 bit integer multiply-add for ~4 and an add, shift
// or logic operation for ~2.  A product of two 64-bit significands is three or
// four multiplies; an exponential is twelve multiplies and some twenty adds and
// shifts, where the FP64 form is nine FP64 operations.  The functions here
// carry 61 or more significant bits through, so each result is rounded once, at
// its end, and is no further from the exact value than the FP64 chain's.
//
// Fixed point: "L" values are base-2 logarithms scaled by 2^52 in a 64-bit
// two's-complement integer (12 integer bits, 52 fraction bits; sums wrap, so
// only a final value has to lie in [-2048, 2048)).  Floating values are a 64-bit
// significand with the top bit set and an exponent of their own.
//
// Plain C++ (the host compiler takes it too, for tests on the CPU).
#pragma once
#include <stdint.h>
#include <string.h>

#include "fx_table.h"

#ifdef __CUDACC__
#define RK_FX __host__ __device__ __forceinline__
#define RK_FX_RARE static __host__ __device__ __noinline__
#else
#define RK_FX inline
#define RK_FX_RARE inline
#endif

namespace rk {
namespace fx {

RK_FX uint64_t mulw(uint32_t a, uint32_t b) { return (uint64_t)a * b; }
RK_FX uint32_t mulh(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
// floor(a b / 2^64) exactly, and less the low halves' product (at most 3 below)
RK_FX uint64_t mulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
RK_FX uint64_t mulhi3(uint64_t a, uint64_t b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
  return mulw(ah, bh) + mulh(ah, bl) + mulh(al, bh);
}
RK_FX int clz(uint64_t x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return __builtin_clzll(x);
#endif
}
RK_FX uint32_t hi32(double x) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__double2hiint(x);
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return (uint32_t)(b >> 32);
#endif
}
RK_FX uint64_t bits_of(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
RK_FX double from_bits(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
// a normal double's significand with the top bit set: |x| = sig 2^(e - 1086),
// e its biased exponent
RK_FX uint64_t significand(double x) { return (bits_of(x) << 11) | 0x8000000000000000ull; }

// 2^f scaled by 2^63 for the fraction f = F 2^-64: 2^(j/256) from the table,
// e^y - 1 by its Taylor polynomial through y^5 for y = r ln2 < 0.00271 (the rest
// is below 2^-60): y to 64 bits, y^2/2 to 48, the tail in 32-bit steps.
// Truncations sum to less than 2^-56 of the result.
RK_FX uint64_t exp2_frac(uint64_t F, const uint64_t* __restrict__ tab) {
  const uint64_t R = F << 8;  // r 2^72: the bits below the table index
  const uint32_t Rh = (uint32_t)(R >> 32), Rl = (uint32_t)R;
  const uint64_t Y = mulw(Rh, RK_FX_LN2_HI) + mulh(Rh, RK_FX_LN2_LO) + mulh(Rl, RK_FX_LN2_HI);  // y 2^72
  const uint32_t yh = (uint32_t)(Y >> 32), yl = (uint32_t)Y;                                    // yh: y 2^40
  const uint64_t Y2 = mulw(yh, yh) + ((uint64_t)mulh(yh, yl) << 1);                             // y^2 2^80
  const uint32_t y2h = (uint32_t)(Y2 >> 32);                                                    // y^2 2^48
  // 1/6 + y/24 + y^2/120 scaled by 2^32, then y^3 times it scaled by 2^88
  const uint32_t c = 0x2aaaaaabu + mulh(yh, 699051u) + mulh(y2h, 546u);
  const uint64_t tail = mulw(mulh(y2h, yh), c);
  const uint64_t P = Y + (Y2 >> 9) + (tail >> 16);  // (e^y - 1) 2^72
  const uint64_t T = tab[(uint32_t)(F >> 56)];
  return T + (mulhi3(T, P) >> 8);
}
// the same for the fraction of L (its low 52 bits), and the floor of L
RK_FX uint64_t exp2_sig(uint64_t L, const uint64_t* __restrict__ tab) { return exp2_frac(L << 12, tab); }
RK_FX int exponent(uint64_t L) { return (int)(uint32_t)(L >> 32) >> 20; }  // floor of the logarithm

// 2^L as a double; the result's exponent must be a normal one (|floor L| <= 1021)
RK_FX double exp2_double(uint64_t L, const uint64_t* __restrict__ tab) {
  const uint64_t m = exp2_sig(L, tab);
  return from_bits(((uint64_t)(uint32_t)(exponent(L) + 1022) << 52) + ((m + 0x400u) >> 11));
}
// the same from a significand and exponent, with 0 below the normal range
RK_FX double pack(uint64_t m, int n) {
  return n < -1021 ? 0.0 : from_bits(((uint64_t)(uint32_t)(n + 1022) << 52) + ((m + 0x400u) >> 11));
}

// exp(x) for |x| < 708
RK_FX double exp_double(double x, const uint64_t* __restrict__ tab) {
  const uint32_t h = hi32(x);
  const int s = 1085 - (int)((h >> 20) & 0x7ffu);  // |x| log2 e = P 2^-s
  const uint64_t P = mulhi(significand(x), RK_FX_LOG2E);
  uint32_t n = 0;
  uint64_t F = 0;
  if (s < 64) {
    n = (uint32_t)(P >> s);
    F = P << (64 - s);
  } else if (s < 128) {
    F = P >> (s - 64);
  }
  if (h >> 31) {  // -(n + F): two's complement over both words
    n = ~n + (F == 0 ? 1u : 0u);
    F = 0ull - F;
  }
  const uint64_t m = exp2_frac(F, tab);
  // (m + 2^10) >> 11 in two steps: m may lie within 2^10 of 2^64
  return from_bits(((uint64_t)(n + 1022u) << 52) + (((m >> 10) + 1u) >> 1));
}

// x log2(e) 2^52 rounded, for |x| < 1400
RK_FX uint64_t log2e_fixed(double x) {
  const uint32_t h = hi32(x);
  const int s = 1033 - (int)((h >> 20) & 0x7ffu);  // the product is P 2^(e - 1085)
  if (s > 63) return 0;
  const uint64_t P = mulhi3(significand(x), RK_FX_LOG2E);
  const uint64_t v = s > 0 ? ((P >> (s - 1)) + 1u) >> 1 : P;
  return (h >> 31) ? 0ull - v : v;
}

// (m 2^(n - 63)) D for a subnormal D (not zero) or a result below the normal range:
// D normalised, the result rounded once where its last place is
RK_FX_RARE double mul_sig_small(uint64_t m, int n, double D) {
  const uint64_t b = bits_of(D), f = b & 0x000fffffffffffffull;
  const int ex = (int)((b >> 52) & 0x7ffu), z = ex == 0 ? clz(f) : 11;
  const uint64_t P0 = mulhi3(m, ex == 0 ? f << z : significand(D));
  const bool top = (P0 >> 63) != 0;
  const uint64_t P = top ? P0 : P0 << 1;
  const int E = n + (ex == 0 ? 12 - z : ex) + (top ? 1 : 0);  // biased exponent, 1 or more if normal
  const int s = E >= 1 ? 11 : 12 - E;                         // bits of P below the last place
  const uint64_t r = s > 64 ? 0ull : ((P >> (s - 1)) + 1u) >> 1;
  const uint64_t q = E >= 2047 ? 0x7ff0000000000000ull : (E >= 1 ? ((uint64_t)(uint32_t)(E - 1) << 52) + r : r);
  return from_bits(q | (b & 0x8000000000000000ull));
}
// (m 2^(n - 63)) D rounded to a double; infinite and NaN D are returned as they are
RK_FX double mul_sig(uint64_t m, int n, double D) {
  const uint32_t h = hi32(D);
  const int eD = (int)((h >> 20) & 0x7ffu);
  const uint64_t P = mulhi3(m, significand(D));  // in [2^62, 2^64)
  const bool top = (P >> 63) != 0;
  const uint64_t r = top ? (P + 0x400u) >> 11 : (P + 0x200u) >> 10;  // 53 bits, or 2^53 after a carry
  const int e = n + eD + (top ? 1 : 0) - 1;
  uint64_t b = ((uint64_t)(uint32_t)e << 52) + r;
  b = e >= 2046 ? 0x7ff0000000000000ull : b;
  if (eD == 0 || e < 0) {
    if (eD != 0x7ff && (bits_of(D) << 1) != 0) return mul_sig_small(m, n, D);
    b = 0ull;
  }
  b |= (uint64_t)(h & 0x80000000u) << 32;
  return from_bits(eD == 0x7ff ? bits_of(D) : b);
}

// ---- sums in 128-bit fixed point.  A set of doubles with largest biased
// exponent em is put on one grid of 2^(hb + em - 1149), hb bits of headroom for
// the sums: each value keeps the bits above 2^-(126 - hb) of the largest (all of its
// 53 down to 2^-(73 - hb) of the largest, fewer below; what is cut is cut downwards,
// at most one unit of the grid), and sums of them are exact in any order and cost
// integer adds.  A sum of values that all lie far below the largest is the caller's to
// form otherwise.
struct Wide {
  uint64_t hi, lo;  // two's complement
};
// infinite and NaN values are the caller's to exclude; subnormal ones become zero
RK_FX Wide to_grid(double x, int em, int hb) {
  const uint32_t h = hi32(x);
  const int e = (int)((h >> 20) & 0x7ffu);
  const uint64_t M = e == 0 ? 0ull : significand(x) >> 1;
  const int64_t V = (int64_t)((h >> 31) ? 0ull - M : M);
  const int s = hb + em - e;  // >= hb >= 1; the value is V 2^64 >> s
  const int s0 = s < 63 ? s : 63, s1 = s < 64 ? 0 : (s < 127 ? s - 64 : 63);
  Wide w;
  w.hi = (uint64_t)(V >> s0);
  w.lo = s < 64 ? (uint64_t)V << (64 - s) : (uint64_t)(V >> s1);
  return w;
}
RK_FX void add(Wide& a, uint64_t hi, uint64_t lo) {
#ifdef __CUDA_ARCH__
  asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;" : "+l"(a.lo), "+l"(a.hi) : "l"(lo), "l"(hi));
#else
  a.lo += lo;
  a.hi += hi + (a.lo < lo ? 1u : 0u);
#endif
}
RK_FX void sub(Wide& a, uint64_t hi, uint64_t lo) {
#ifdef __CUDA_ARCH__
  asm("sub.cc.u64 %0, %0, %2;\n\tsubc.u64 %1, %1, %3;" : "+l"(a.lo), "+l"(a.hi) : "l"(lo), "l"(hi));
#else
  const uint64_t l = a.lo;
  a.lo -= lo;
  a.hi -= hi + (l < lo ? 1u : 0u);
#endif
}
// a 2^(hb + em - 1149) rounded to a double (zero below the normal range; it must not
// lie above, which em + hb < 2047 ensures)
RK_FX double from_grid(Wide a, int em, int hb) {
  const uint64_t neg = 0ull - (a.hi >> 63);  // all ones if negative
  const uint64_t lo = (a.lo ^ neg) - neg;
  const uint64_t hi = (a.hi ^ neg) + (neg && lo == 0 ? 1u : 0u);
  const bool up = hi != 0;
  const uint64_t w1 = up ? hi : lo, w0 = up ? lo : 0;
  const int z = w1 ? clz(w1) : 0;
  const uint64_t top = (w1 << z) | ((w0 >> 1) >> (63 - z));
  const int E = hb + em + 1 - z - (up ? 0 : 64);
  const uint64_t b = ((uint64_t)(uint32_t)(E - 1) << 52) + (((top >> 10) + 1u) >> 1);
  return from_bits((E <= 0 || w1 == 0 ? 0ull : b) | (neg << 63));
}

// The fixed-point Arrhenius form: log2 k = log2 A + b log2 T - (Ea / R) log2 e / T.
// Coefficients are stored shifted to be non-negative (b + 32 scaled by 2^57, Ea/R
// log2 e + 2^15 scaled by 2^46), the shifts taken out once per cell.
// Valid for |b| <= 16, Ea/R log2 e in [-2^13, 130000), |log2 A| <= 150 and T in
// [T_LO, T_HI): a rate constant's logarithm (between -1242 and 429) and those of two
// Gibbs factors (each below 246 in magnitude) then stay inside (-1735, 922), which
// neither wraps nor overflows a double.  A mechanism's own lowest temperature may be
// higher: where its slowest rate constant passes 2^-500, so that kappa stays normal.
constexpr double T_LO = 150.0, T_HI = 16000.0;
struct Temp {
  uint64_t lgT, iT, c;  // log2 T 2^59, 2^70 / T, and the shifts' share
};
// log2 x 2^59 for normal x >= 1 (Tang's table-driven method): x = 2^e m, r = m /
// c_j - 1 with |r| <= 2^-8, ln(1 + r) through r^7; 2^-55 absolute, where the FP64
// form ends with half an ulp of ln T (4e-16) and takes eleven FP64 instructions.
RK_FX uint64_t log2_fixed(double x, const uint64_t* __restrict__ inv_c, const uint64_t* __restrict__ log2_c) {
  const uint64_t M = significand(x);
  const int j = (int)(M >> 56) & 127;
  const int64_t r = (int64_t)(mulhi(M, inv_c[j]) - 0x8000000000000000ull);  // r 2^63
  const bool neg = r < 0;
  const uint64_t R = (uint64_t)(neg ? -r : r) << 8;  // |r| 2^71
  const uint32_t rh = (uint32_t)(R >> 32);           // |r| 2^39
  const uint64_t r2 = mulhi3(R, R);                  // r^2 2^78
  const uint32_t r2h = (uint32_t)(r2 >> 30);         // r^2 2^48
  const uint64_t r3 = mulw(r2h, rh);                 // |r|^3 2^87
  // c = 1/3 - r/4 + r^2/5 - r^3/6 scaled by 2^32 (r^4/7 is below one unit)
  const uint32_t c1 = rh >> 9, c2 = (r2h >> 16) / 5u, c3 = (uint32_t)(r3 >> 55) / 6u;
  const uint32_t c = neg ? 0x55555557u + c1 + c2 + c3 : 0x55555555u - c1 + c2 - c3;
  const uint64_t t = mulw((uint32_t)(r3 >> 32), c) + mulh((uint32_t)r3, c);  // |r|^3 c 2^87
  const uint64_t odd = R + (t >> 16), sq = r2 >> 8;                          // scaled by 2^71
  const uint64_t mag = neg ? odd + sq : odd - sq;
  const uint64_t lg = mulhi(mag, RK_FX_LOG2E) >> 11;  // |log2(1 + r)| 2^59
  const uint64_t base = log2_c[j] + ((uint64_t)(uint32_t)((int)((hi32(x) >> 20) & 0x7ffu) - 1023) << 59);
  return neg ? base - lg : base + lg;
}
// v 2^-59 as a double, for v >= 2^59
RK_FX double from_fixed59(uint64_t v) {
  const int z = clz(v);
  v <<= z;
  return from_bits(((uint64_t)(uint32_t)(1023 + 4 - z - 1) << 52) + (((v >> 10) + 1u) >> 1));
}
// 2^70 / T from T and its reciprocal rounded to a double: the residual T r - 1 is
// formed in 128 bits and taken off
RK_FX uint64_t recip_fixed70(double T, double invT) {
  const uint64_t M = significand(T), y = significand(invT);
  // M y = 2^126 (1 + d) or 2^127 (1 + d), |d| < 2^-51
  const uint64_t hi = mulhi(M, y), lo = M * y;
  const uint64_t one = (hi + (1ull << 40)) & ~((1ull << 41) - 1);  // 2^62 or 2^63
  const int64_t d = (int64_t)(((hi - one) << 32) | (lo >> 32));    // d 2^94 or 2^95
  const int up = one >> 63 ? 1 : 0;
  const int64_t corr = ((int64_t)(y >> 32) * (d >> 18)) >> (44 + up);
  const int sh = 1016 - (int)((hi32(invT) >> 20) & 0x7ffu);
  return (y >> sh) - (uint64_t)(corr >> sh);
}
RK_FX Temp temperature(uint64_t lgT, uint64_t iT) {
  Temp t;
  t.lgT = lgT;
  t.iT = iT;
  t.c = (t.iT >> 3) - (t.lgT >> 2);
  return t;
}
RK_FX uint64_t arrhenius(const Temp& t, uint64_t lgA, uint64_t b, uint64_t E) {
  return lgA + mulhi(b, t.lgT) - mulhi(E, t.iT) + t.c;
}

}  // namespace fx
}  // namespace rk
