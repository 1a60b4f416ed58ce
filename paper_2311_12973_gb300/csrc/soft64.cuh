// soft64.cuh -- FP64-accurate functions of the particle filter on the integer pipe.
//
// GB300's FP64 pipe retires 1.65 lanes per clock and SM (measured; add, multiply and
// FMA alike, conversions 1.95) against 128 for integer and FP32 instructions, so one
// FP64 instruction takes the time of 78 others.  An FP64 filter step written with the
// math library runs about 150 of them per particle.  The functions below evaluate the
// same quantities in 64-bit fixed point: a high product of two 64-bit integers is 19
// issue slots, a whole exponential about 100, a pair of Box-Muller normals about 450,
// where the library's run 17 and 90 FP64 instructions.  Each is a table reduction
// followed by a short power series (2^(i/256) and 2^(i/65536) for the exponential;
// ln of 256 cells for the logarithm; cos and sin at multiples of pi/1024 with the
// angle-addition formulas; one Halley step for the square root), with every stage
// carried to 2^-60 or better.  What that leaves: the exponential is within 2^-56
// relative before its use, log1p(x) - x next to 0 within half an ulp of x, and a
// normal within 1.5 ulp (next to a zero of its sine the angle's absolute 2^-64
// counts; largest seen 1.31 over 6 10^7, root mean square 0.29, 0.7 % beyond
// 0.52; the library's log and sincospi are within 1 ulp each).
//
// Fixed-point notation: "Qk" is an integer holding value 2^k.
#pragma once

#include <cstdint>
#include <cstring>

#include "soft64_tables.h"

#ifdef __CUDACC__
#define S64_FN __host__ __device__ __forceinline__
#else
#include <cmath>
#define S64_FN inline
#endif

namespace smc2 {

S64_FN uint64_t s64_mulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
S64_FN uint32_t s64_mulhi32(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
S64_FN int s64_mulhi32s(int a, int b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int)(((int64_t)a * b) >> 32);
#endif
}
// leading zeros of v >= 2^32, by the exponent of the high word's conversion to float (rounded
// towards zero): the conversion runs at 62 lanes per clock and SM, the leading-bit search at 16
S64_FN int s64_clz(uint64_t v) {
#ifdef __CUDA_ARCH__
  return 158 - (int)(__float_as_uint(__uint2float_rz((uint32_t)(v >> 32))) >> 23);
#else
  return __builtin_clzll(v);
#endif
}
S64_FN uint64_t s64_bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
S64_FN double s64_double(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
S64_FN uint32_t s64_float_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  memcpy(&b, &x, 4);
  return b;
#endif
}
S64_FN float s64_rsqrt(float x) {  // 1/sqrt(x) to about 2^-22
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / sqrtf(x);
#endif
}

// Kernels read the tables (g_soft64) from a copy in shared memory where it has room: a
// warp's lanes read unrelated entries, which costs a shared load a few bank conflicts and a
// cached global load one pass per cache line (up to 32).

// ---------------------------------------------------------------------------
// packing
// ---------------------------------------------------------------------------
// mantissa (leading one at bit 63; 0 for a zero or subnormal x) and exponent of a
// finite x >= 0: x = m 2^(e - 63)
S64_FN uint64_t s64_unpack(double x, int& e) {
  const uint64_t b = s64_bits(x);
  const uint32_t ef = (uint32_t)(b >> 52);
  e = (int)ef - 1023;
  return ef ? (b << 11) | 0x8000000000000000ull : 0ull;
}
// p 2^(e - 62) as a double, p in [2^62, 2^63], rounded to nearest (ties up); e a normal exponent
S64_FN double s64_pack62(uint64_t p, int e) {
  return s64_double(((uint64_t)(uint32_t)(e + 1022) << 52) + (p >> 10) + ((p >> 9) & 1ull));
}

// ---------------------------------------------------------------------------
// exponential
// ---------------------------------------------------------------------------
// signed Q57 of x, |x| < 64 (truncated towards zero)
S64_FN int64_t s64_q57(double x) {
  const uint64_t b = s64_bits(x);
  const uint32_t s = 1023u + 6u - ((uint32_t)(b >> 52) & 0x7ffu);  // right shift of the mantissa at bit 63
  const uint64_t v = s > 63u ? 0ull : ((b << 11) | 0x8000000000000000ull) >> s;
  return (int64_t)b < 0 ? -(int64_t)v : (int64_t)v;
}
// e^(X 2^-57) = m 2^(k - 61), m within a 2^-15 part of [2^61, 2^62], relative error below 2^-57
// (the truncation of the argument's Q57).  X = k ln 2 + j ln 2 / 65536 + r; 2^(j / 65536)
// from two tables, e^r = 1 + r + r^2/2 + r^3/6.
S64_FN uint64_t s64_exp_q57(int64_t X, const Soft64Tables& T, int& k) {
  const int i = s64_mulhi32s((int)(X >> 32), 12102203);  // X 65536 / ln 2, to one unit
  k = i >> 16;
  const uint32_t j = (uint32_t)i & 0xffffu;
  const int64_t r = (int64_t)(((uint64_t)X << 18) - (uint64_t)(int64_t)k * kLn2Q75 - (uint64_t)j * kStepQ75);  // Q75
  const int rh = (int)(r >> 29);                             // Q46
  const int r2 = s64_mulhi32s(rh, rh);                       // r^2 in Q60
  const int r3 = s64_mulhi32s(s64_mulhi32s(r2, rh), 0x55555555);  // r^3 / 3 in Q74
  const uint64_t F = 0x8000000000000000ull + (uint64_t)(r >> 12) + ((uint64_t)(int64_t)(r2 + (r3 >> 14)) << 2);  // Q63
  return s64_mulhi(s64_mulhi(T.exp1[j >> 8], T.exp2[j & 255u]), F);
}

// ---------------------------------------------------------------------------
// logarithm
// ---------------------------------------------------------------------------
// r - log1p(r) in Q79 for |r| < 2^-8, r in Q71 and r2 = r^2 in Q78:
// |r| (r/2 - r^2 (1/3 - r/4 + r^2/5 - r^3/6 + r^4/7)), absolute error below 2^-57 |r|
S64_FN uint64_t s64_log1p_tail(int64_t r, uint64_t r2) {
  const uint32_t r2h = (uint32_t)(r2 >> 32);  // Q46
  const uint32_t in = 858993459u - (uint32_t)s64_mulhi32s((int)(r >> 32), 5592405) + s64_mulhi32(r2h, 37449u);  // Q32
  const uint64_t W = 0x5555555555555555ull - (uint64_t)(r >> 9) + ((uint64_t)s64_mulhi32(r2h, in) << 18);       // Q64
  const uint64_t q2 = s64_mulhi(r2, W) >> 6;  // Q72
  const uint64_t ar = (uint64_t)(r < 0 ? -r : r);
  return s64_mulhi(ar, r < 0 ? ar + q2 : ar - q2);
}

// ---------------------------------------------------------------------------
// two normals from two words (Box-Muller): u = (2 (w >> 9) + 1) 2^-24,
// z0 = sqrt(-2 ln u_a) cos(2 pi u_b), z1 the same with sin
// ---------------------------------------------------------------------------
S64_FN uint64_t s64_sqrt_m2ln(uint32_t wa, const Soft64Tables& T, int& h) {  // Q61 in [1, 2], times 2^h
  // -ln u: u = m 2^(e - 24), m a float's mantissa; m I / 2048 = 1 + r exactly (32-bit product, Q34)
  const uint32_t fb = s64_float_bits((float)(((wa >> 9) << 1) | 1u));
  const uint32_t j = (fb >> 15) & 255u;
  const int r32 = (int)(((fb & 0x7fffffu) | 0x800000u) * T.inv[j]);
  const int E = 24 + 127 - (int)(fb >> 23) - (j >= (uint32_t)kLnHalf ? 1 : 0);
  const int64_t r = (int64_t)((uint64_t)(int64_t)r32 << 37);
  const uint64_t q = s64_log1p_tail(r, (uint64_t)((int64_t)r32 * r32) << 10);
  const int64_t b = -(int64_t)T.ln[j] - (r >> 7) + (int64_t)(q >> 15);  // Q64
  uint64_t V = (uint64_t)b;
  int s = 64;
  if (E > 0) {
    V = (uint64_t)E * kLn2Q58 + (uint64_t)(b >> 6);
    s = 58;
  }
  if (E == 0 && j == 255u) {  // next to 1: -ln u = d + q with d = 1 - u exact, at the scale that keeps its digits
    const uint64_t d = (uint64_t)(-r32);
    const bool small = d < (1u << 17);
    V = small ? (d << 46) + (q << 1) : (d << 38) + (q >> 7);
    s = small ? 80 : 72;
  }
  const int lz = s64_clz(V);
  const uint64_t v = V << lz;
  const int t = 64 - lz - s;           // 2 (-ln u) = v 2^(t - 63)
  const uint64_t A = (t & 1) ? v : v >> 1;  // Q62 in [1, 4), times 2^(t - (t & 1))
  h = t >> 1;
  // sqrt(A) = A y (1 + e/2 + 3 e^2 / 8), e = 1 - A y^2, y the float reciprocal square root
  const uint32_t Y = (uint32_t)(s64_rsqrt((float)(uint32_t)(A >> 32) * 0x1p-30f) * 0x1p31f);  // exact
  const int64_t e = (int64_t)(0x2000000000000000ull - s64_mulhi(A, ((uint64_t)Y * Y) << 1));  // Q61
  const int eh = (int)(e >> 10);                                                             // Q51
  const int64_t c = (e >> 1) + (int64_t)((uint32_t)s64_mulhi32s(eh, eh) * 3u >> 12);
  const uint64_t p0 = (A >> 32) * Y + (((A & 0xffffffffull) * Y) >> 32);  // A y, Q61
  const uint64_t ac = (uint64_t)(c < 0 ? -c : c);
  const uint64_t dp = s64_mulhi(p0, ac << 24) >> 21;
  return c < 0 ? p0 - dp : p0 + dp;
}
S64_FN void s64_normal_pair(uint32_t wa, uint32_t wb, const Soft64Tables& T, double& z0, double& z1) {
  int h;
  const uint64_t rho = s64_sqrt_m2ln(wa, T, h) << 2;  // Q63
  // 2 pi u_b = oct pi/4 + phi, phi (or pi/4 - phi in odd octants) = (pi/4) t 2^-21 = A pi/1024 + delta,
  // delta = d (pi/4) 2^-21, |d| <= 4096
  const uint32_t n = ((wb >> 9) << 1) | 1u;
  const uint32_t oct = n >> 21;
  uint32_t t = n & 0x1fffffu;
  t = (oct & 1u) ? 0x200000u - t : t;
  const uint32_t A = (t + 4096u) >> 13;
  const int d = (int)t - (int)(A << 13);
  const uint32_t ad = (uint32_t)(d < 0 ? -d : d), d2 = ad * ad;
  const uint32_t d4 = (d2 >> 9) * (d2 >> 9);
  // sin(delta) = d P, P = K - d^2 K^3/6 + d^4 K^5/120 (Q84)
  const uint64_t P = kSinC1 - (((uint64_t)d2 * (uint32_t)kSinC3) >> 14) + s64_mulhi32(d4, (uint32_t)kSinC5);
  const uint64_t sd = ((uint64_t)ad * (uint32_t)(P >> 32) << 20) + (((uint64_t)ad * (uint32_t)P) >> 12);  // Q72
  // 1 - cos(delta) = d^2 K^2/2 - d^4 K^4/24 (Q72)
  const uint64_t u = (((uint64_t)d2 * (uint32_t)(kCosC2 >> 32)) << 8) + (((uint64_t)d2 * (uint32_t)kCosC2) >> 24) -
                     ((uint64_t)s64_mulhi32(d4, (uint32_t)kCosC4) << 1);
  const uint64_t cA = T.cossin[2 * A], sA = T.cossin[2 * A + 1];  // Q63, Q64
  const uint64_t s2 = s64_mulhi(sA, sd), c2 = s64_mulhi(cA, sd);  // Q72, Q71
  const uint64_t s1 = s64_mulhi(sA, u), c1 = s64_mulhi(cA, u);    // Q72, Q71
  const int64_t ss = d < 0 ? -(int64_t)(s2 >> 1) : (int64_t)(s2 >> 1), cs = d < 0 ? -(int64_t)c2 : (int64_t)c2;
  const uint64_t co = cA - (uint64_t)(((int64_t)c1 + ss) >> 8);      // cos phi, Q63
  uint64_t si = sA + (uint64_t)((cs - (int64_t)(s1 >> 1)) >> 7);     // sin phi, Q64
  int ls;
  if (A == 0) {  // sin phi = d P to all digits
    const int la = s64_clz((uint64_t)ad << 32);
    si = s64_mulhi((uint64_t)ad << (la + 32), P << 1);
    ls = s64_clz(si);
    si <<= ls;
    ls += la - 11;  // ad 2^(la + 32) . P 2 / 2^64 = sin 2^(la + 32 + 84 + 1 - 64)
  } else {
    ls = s64_clz(si);
    si <<= ls;
  }
  uint64_t pc = s64_mulhi(rho, co);  // Q62 in [2^61.5, 2^63]
  int ec = h;
  if (!(pc >> 62)) {
    pc <<= 1;
    --ec;
  }
  uint64_t ps = s64_mulhi(rho, si);  // Q63 in [2^62, 2^64)
  int es = h - ls;
  if (ps >> 63) {
    ps >>= 1;
  } else {
    --es;
  }
  const uint64_t zc = s64_bits(s64_pack62(pc, ec)), zs = s64_bits(s64_pack62(ps, es));
  const bool swap = ((oct + 1u) & 2u) != 0;
  const uint64_t nc = (uint64_t)((oct + 2u) & 4u) << 61, ns = (uint64_t)(oct & 4u) << 61;
  z0 = s64_double((swap ? zs : zc) | nc);
  z1 = s64_double((swap ? zc : zs) | ns);
}

// v 2^-q as a double (either sign, rounded to nearest)
S64_FN double s64_from_fixed(int64_t v, int q) {
  const uint64_t a = (uint64_t)(v < 0 ? -v : v);
  if (a == 0) return 0.0;
  const int lo = (a >> 32) == 0ull ? 32 : 0;
  const int lz = s64_clz(a << lo) + lo;
  const uint64_t b = s64_bits(s64_pack62((a << lz) >> 1, 63 - lz - q));
  return s64_double(b | ((uint64_t)v & 0x8000000000000000ull));
}

// ---------------------------------------------------------------------------
// Poisson log-weight
// ---------------------------------------------------------------------------
// log1p(d) - d for w = 1 + d = lam / y: the arguments are lam > 0 normal and 1/y as its mantissa
// inv_m (64 bits, leading one) and exponent inv_e.  x ln 2 + ln c + log1p(r) - d is formed in
// Q64 for w in about [0.71, 1.42], in the cells next to 1 as the series' tail alone, in Q79, and
// in Q56 for the other w between 2^-60 and 64; outside, ok is false.
S64_FN double s64_log1p_minus(double lam, uint64_t inv_m, int inv_e, const Soft64Tables& T, bool& ok) {
  int x;
  uint64_t W = s64_mulhi(s64_unpack(lam, x), inv_m);  // Q62 in [1, 4)
  x += inv_e;
  if (W >> 63)
    ++x;
  else
    W <<= 1;
  const uint32_t j = (uint32_t)(W >> 55) & 255u;
  const bool half = j >= (uint32_t)kLnHalf;
  const int xx = x + (half ? 1 : 0);
  const uint32_t I = T.inv[j];
  const uint64_t lo = (W & 0xffffffffull) * I, hi = (W >> 32) * I + (lo >> 32);
  const int64_t r = (int64_t)((hi << 29) | ((lo & 0xffffffffull) >> 3));  // Q71 of W I / 2^11 - 1
  const uint64_t ar = (uint64_t)(r < 0 ? -r : r);
  const uint64_t q = s64_log1p_tail(r, s64_mulhi(ar, ar));
  const int64_t b = (int64_t)T.ln[j] + (r >> 7) - (int64_t)(q >> 15);  // ln of the reduced argument, Q64
  ok = x <= 5 && x >= -60;
  int64_t v = b - (int64_t)(half ? W : (W << 1));  // less d = W - 1 (Q64: W 2^63 or 2^64 at one)
  int qs = 64;
  if (j == 0u || j == 255u) {
    v = -(int64_t)q;
    qs = 79;
  }
  if (xx != 0) {
    const uint32_t sh = (uint32_t)(7 - x);
    v = (int64_t)xx * (int64_t)kLn2Q56 + (b >> 8) + (int64_t)(1ull << 56) - (int64_t)(W >> (sh > 63u ? 63u : sh));
    qs = 56;
  }
  return s64_from_fixed(v, qs);
}

}  // namespace smc2
