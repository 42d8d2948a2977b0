// Fixed-point complex logarithm and exponential for the FP64 kernels (host and
// device).  The FP64 pipe of sm_103a takes two lanes a clock per SM, 1/64 of
// the FP32 rate, so a warp-wide FP64 instruction costs as much as 64 issue
// slots, and the CUDA library's log, atan2, exp and sincos run on that pipe.
// Here they run on the integer pipe, in 64-bit fixed point:
//
//   log:  y -> (log2|y| modulo 16 in units of 2^-60, arg y in units of 2^-64
//         revolution, log2|y| in FP32).  An exponent sum <a, log y> is then
//         integer arithmetic: the phase is exact modulo one revolution, and
//         the FP32 sum supplies the integer part that the 64-bit sum lost.
//   exp:  2^W (cos, sin)(2 pi theta) as two 62-bit fractions and a power of
//         two, rounded once to double.
//
// Both are table lookups followed by a short polynomial: exp2 and sincos by
// Tang's table-driven method (P. T. P. Tang, "Table-driven implementation of
// the exponential function in IEEE floating-point arithmetic", ACM TOMS 15,
// 1989) with two tables of 64 entries, log2 by his method for the logarithm
// (ACM TOMS 16, 1990) with 128 entries, the angle by the addition theorem of
// atan with tan(alpha_i) = i/32.  The tables are computed by the compiler
// from Taylor series, repeated squaring and Euler's series, in 128-bit
// integers.  Largest errors over a million random arguments, against 113 bits:
// 2^-58.5 in log2|y|, 2^-59.7 revolution in the angle, 2^-57.7 in cos and sin,
// 2^-57.2 in exp2 (of values up to 2); what is exact: phases of whole quarter
// turns (points on the axes) and their cos and sin.
//
// Qn below means a fixed-point number with n fraction bits.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define HPT_FX __host__ __device__ __forceinline__
#else
#define HPT_FX inline
#endif

namespace hpt {
namespace fx {

typedef unsigned __int128 u128;

struct Tables {
  int64_t exp1[64];       // 2^(i/64), Q62
  int64_t exp2[64];       // 2^((j + 1/2)/4096), Q62
  int64_t cs1[64][2];     // cos, sin of i/64 revolution, Q62
  int64_t cs2[64][2];     // cos, sin of j/4096 revolution, Q62
  uint64_t at[33];        // atan(i/32) in revolutions, Q64
  int64_t lat[33];        // log2 sqrt(1 + (i/32)^2), Q60
  uint32_t rcp[128];      // 1/(1 + (i + 1/2)/128), Q32
  int64_t lrcp[128];      // -log2 of rcp[i]/2^32, Q60
};

// ---- the tables, at compile time -------------------------------------------
// Q90 numbers in 128 bits (values below 2^10).
constexpr u128 mul90(u128 a, u128 b) {
  const u128 m = ((u128)1 << 46) - 1;
  const u128 ah = a >> 46, al = a & m, bh = b >> 46, bl = b & m;
  return ((ah * bh) << 2) + ((ah * bl + al * bh) >> 44) + ((al * bl) >> 90);
}
constexpr u128 kPi90 = ((u128)0xc90fdaaull << 64) | 0x22168c234c4c6629ull;
constexpr u128 kLn2_90 = ((u128)0x2c5c85full << 64) | 0xdf473de6af278eceull;
constexpr u128 kOne90 = (u128)1 << 90;
constexpr int64_t round90(u128 v, int q) { return (int64_t)((v + ((u128)1 << (89 - q))) >> (90 - q)); }

constexpr u128 exp90(u128 x) {   // Taylor, 0 <= x < 1
  u128 term = kOne90, sum = kOne90;
  for (int i = 1; i < 30; ++i) {
    term = mul90(term, x) / (unsigned)i;
    sum += term;
  }
  return sum;
}
// Taylor series of cos (first = 0) or sin (first = 1) of 0 <= x < 2 pi, Q62
constexpr int64_t cs62(u128 x, int first) {
  u128 term = kOne90, pos = 0, neg = 0;
  for (int i = 0; i < 46; ++i) {
    if ((i & 1) == first) {
      if (((i >> 1) & 1) == 0) pos += term;
      else neg += term;
    }
    term = mul90(term, x) / (unsigned)(i + 1);
  }
  return pos >= neg ? round90(pos - neg, 62) : -round90(neg - pos, 62);
}
constexpr int64_t log2_60(u128 x) {   // 1 <= x < 2, Q60, by repeated squaring
  u128 r = 0;
  for (int b = 0; b < 64; ++b) {
    x = mul90(x, x);
    r <<= 1;
    if (x >= 2 * kOne90) {
      r |= 1;
      x >>= 1;
    }
  }
  return (int64_t)((r + 8) >> 4);
}
constexpr u128 atan90(int i) {   // atan(i/32) by Euler's series (ratio at most 1/2)
  if (i == 0) return 0;
  const unsigned d = 1024 + (unsigned)(i * i);
  u128 term = kOne90 * (unsigned)(32 * i) / d, sum = 0;
  for (int k = 0; k < 96; ++k) {
    sum += term;
    term = term * (unsigned)(i * i * (2 * k + 2)) / (d * (unsigned)(2 * k + 3));
  }
  return sum;
}
constexpr Tables make_tables() {
  Tables t{};
  for (int i = 0; i < 64; ++i) {
    t.exp1[i] = round90(exp90(kLn2_90 * (unsigned)i / 64), 62);
    t.exp2[i] = round90(exp90(kLn2_90 * (unsigned)(2 * i + 1) / 8192), 62);
    const u128 x1 = kPi90 * (unsigned)i / 32, x2 = kPi90 * (unsigned)i / 2048;
    t.cs1[i][0] = cs62(x1, 0);
    t.cs1[i][1] = cs62(x1, 1);
    t.cs2[i][0] = cs62(x2, 0);
    t.cs2[i][1] = cs62(x2, 1);
  }
  for (int i = 0; i <= 32; ++i) {
    // atan / (2 pi): the quotient bit by bit, Q64
    u128 a = atan90(i), q = 0;
    const u128 tp = 2 * kPi90;
    for (int b = 0; b < 65; ++b) {
      a <<= 1;
      q <<= 1;
      if (a >= tp) {
        a -= tp;
        q |= 1;
      }
    }
    t.at[i] = (uint64_t)((q + 1) >> 1);
    t.lat[i] = i == 32 ? (int64_t)1 << 59 : log2_60(kOne90 + (kOne90 >> 10) * (unsigned)(i * i)) / 2;
  }
  for (int i = 0; i < 128; ++i) {
    t.rcp[i] = (uint32_t)((((uint64_t)1 << 40) + (257 + 2 * i) / 2) / (unsigned)(257 + 2 * i));
    t.lrcp[i] = ((int64_t)1 << 60) - log2_60((u128)t.rcp[i] << 59);
  }
  return t;
}

#ifdef __CUDACC__
static __device__ const Tables d_tables = make_tables();
#endif
static constexpr Tables h_tables = make_tables();
HPT_FX const Tables& tables() {
#ifdef __CUDA_ARCH__
  return d_tables;
#else
  return h_tables;
#endif
}

// ---- arithmetic ---------------------------------------------------------------
// a b / 2^62 for |a|, |b| < 2^63 with |a b| < 2^125, within about four units:
// three 32 x 32 -> 64-bit products (the low halves' product is left out).
HPT_FX int64_t mul62(int64_t a, int64_t b) {
  const int32_t ah = (int32_t)(a >> 32), bh = (int32_t)(b >> 32);
  const int32_t al = (int32_t)((uint32_t)a >> 1), bl = (int32_t)((uint32_t)b >> 1);
  return (int64_t)((uint64_t)((int64_t)ah * bh) << 2) + (((int64_t)ah * bl + (int64_t)al * bh) >> 29);
}
HPT_FX int32_t mulhi32(int32_t a, int32_t b) { return (int32_t)(((int64_t)a * b) >> 32); }
HPT_FX int clz64(uint64_t v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return v ? __builtin_clzll(v) : 64;
#endif
}
HPT_FX uint64_t bits_of(double v) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(v);
#else
  uint64_t b;
  memcpy(&b, &v, 8);
  return b;
#endif
}
HPT_FX double of_bits(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double v;
  memcpy(&v, &b, 8);
  return v;
#endif
}
HPT_FX float rcp_f(float v) {
#ifdef __CUDA_ARCH__
  return __frcp_rn(v);
#else
  return 1.0f / v;
#endif
}

struct Log {
  int64_t l;      // log2|y| modulo 16, Q60
  uint64_t turn;  // arg y / (2 pi) modulo 1, Q64
  float lf;       // log2|y|
};

// The logarithm of y = (re, im).  Returns false for y = 0, infinities and NaN
// (out then holds zeros).
HPT_FX bool log_of(double re, double im, Log& out) {
  const Tables& T = tables();
  const uint64_t mant = ((uint64_t)1 << 52) - 1;
  const uint64_t br = bits_of(re) & ~((uint64_t)1 << 63), bi = bits_of(im) & ~((uint64_t)1 << 63);
  const bool swap = br < bi;
  const uint64_t ba = swap ? bi : br, bb = swap ? br : bi;   // |larger|, |smaller|
  out.l = 0;
  out.turn = 0;
  out.lf = 0.f;
  int ea = (int)(ba >> 52), eb = (int)(bb >> 52);
  if (ea == 0x7ff || ba == 0) return false;
  // a in [2^57, 2^58), b on the same scale, rounded to its last bit
  uint64_t ma = ea ? (ba & mant) | (mant + 1) : ba, mb = eb ? (bb & mant) | (mant + 1) : bb;
  ea = ea ? ea : 1;
  eb = eb ? eb : 1;
  if (ma <= mant) {   // both subnormal
    const int s = clz64(ma) - 11;
    ma <<= s;
    mb <<= s;
    ea -= s;
    eb -= s;
  }
  const int d = ea - eb;
  const uint64_t A = ma << 5;
  const uint64_t B = d < 60 ? (((mb << 6) >> d) + 1) >> 1 : 0;
  // rotate by -atan(i/32): exact integers, tangent of what is left at most 1/64
  const float rf = (float)(uint32_t)(B >> 32) * rcp_f((float)(uint32_t)(A >> 32));
  int i = (int)(rf * 32.f + 0.5f);
  i = i > 32 ? 32 : i;
  uint64_t a = (A << 5) + B * (uint32_t)i;
  int64_t b = (int64_t)(B << 5) - (int64_t)(A * (uint32_t)i);
  const int es = a >> 63 ? 0 : 1;   // a in [2^63, 2^64)
  a <<= es;
  b = (int64_t)((uint64_t)b << es);
  // u = b / a, Q67: reciprocal from FP32, one Newton step, one residual
  const uint32_t r0 = (uint32_t)(rcp_f((float)(uint32_t)(a >> 32)) * 4611686018427387904.f);
  const uint64_t P = (a >> 32) * r0 + (((a & 0xffffffffu) * r0) >> 32);
  const int64_t E = (int64_t)(((uint64_t)1 << 62) - P);
  uint64_t r1 = ((uint64_t)r0 << 32) + (uint64_t)(((int64_t)r0 * (int32_t)(E >> 12)) >> 18);
  r1 = r1 >> 63 ? ~((uint64_t)1 << 63) : r1;
  const int64_t u0 = (int64_t)((uint64_t)mul62(b, (int64_t)r1) << 3);
  const int64_t rem = (int64_t)((uint64_t)b << 4) - mul62(u0, (int64_t)(a >> 1));
  const int64_t u = u0 + ((rem * (int64_t)r0) >> 31);
  const int64_t v = mul62(u, u);   // u^2, Q72
  const int32_t v32 = (int32_t)(v >> 30);                        // Q42
  const int32_t vv = (int32_t)(((int64_t)v32 * v32) >> 32);      // u^4, Q52
  // atan(u)/(2 pi) = u (1 - v/3 + v^2 (1/5 - v/7 + v^2/9)) / (2 pi)
  const int32_t t7 = 0x2e906eb - (mulhi32(v32, 0x2437729) >> 10);
  const int32_t t5 = 0x41309b0 - (mulhi32(v32, t7) >> 10);
  const int64_t pa = 0xa2f9836e4e44153ll - (mul62(v, 0x36532bcf6f6c071ll) >> 10) + (((int64_t)vv * t5) >> 21);
  uint64_t th = T.at[i] + (uint64_t)(mul62(u, pa) >> 3);
  if (swap) th = ((uint64_t)1 << 62) - th;
  if (bits_of(re) >> 63) th = ((uint64_t)1 << 63) - th;
  if (bits_of(im) >> 63) th = 0 - th;
  // log2 sqrt(1 + v) = v (1/2 - v/4 + v^2/6 - v^3/8) / ln 2
  const int32_t h3 = 0x1ec709dc - (mulhi32(v32, 0x17154765) >> 10);
  const int64_t w = 0x2e2a8eca5705fc2fll - (mul62(v, 0x171547652b82fe17ll) >> 10) + (((int64_t)vv * h3) >> 21);
  const int64_t lg1 = mul62(v, w) >> 12;
  // log2(a / 2^63) = log2(1 + x) - log2 c, x = a c - 1, |x| <= 2^-8
  const int k = (int)(a >> 56) & 127;
  const uint32_t c = T.rcp[k];
  const int64_t x63 = (int64_t)(((a >> 32) * c + (((a & 0xffffffffu) * c) >> 32)) - ((uint64_t)1 << 63));
  const int64_t x = (int64_t)((uint64_t)x63 << 5);   // Q68
  const int32_t x32 = (int32_t)(x63 >> 25);          // Q38
  const int32_t s6 = 0x1ec709dc - (mulhi32(x32, 0x1a61762a) >> 6);
  const int32_t s5 = 0x24eed8a2 - (mulhi32(x32, s6) >> 6);
  const int32_t s4 = 0x2e2a8eca - (mulhi32(x32, s5) >> 6);
  const int64_t y3 = 0x1ec709dc3a03fd75ll - (((int64_t)x32 * s4) >> 7);
  const int64_t y2 = 0x2e2a8eca5705fc2fll - (mul62(x, y3) >> 6);
  const int64_t y1 = 0x5c551d94ae0bf85ell - (mul62(x, y2) >> 6);
  const int64_t frac = (mul62(x, y1) >> 8) + T.lrcp[k] - T.lat[i] + lg1;
  const int e = ea - 1022 - es;
  out.l = (int64_t)(((uint64_t)(int64_t)e << 60) + (uint64_t)frac);
  out.turn = th;
  out.lf = (float)e + (float)(int32_t)(frac >> 32) * 3.7252902984619140625e-9f;   // 2^-28
  return true;
}

// t log2(e), modulo 16, as a 128-bit fraction (Q124: hi Q60, lo the next 64
// bits), for exponent sums that multiply it by large integers.  t finite.
struct Wide {
  uint64_t hi, lo;
};
HPT_FX uint64_t umulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((u128)a * b) >> 64);
#endif
}
HPT_FX Wide log2e_times(double t) {
  const uint64_t bt = bits_of(t), mag = bt & ~((uint64_t)1 << 63);
  const int e = (int)(mag >> 52) ? (int)(mag >> 52) : 1;
  const uint64_t m = ((mag >> 52) ? (mag & (((uint64_t)1 << 52) - 1)) | ((uint64_t)1 << 52) : mag) << 11;   // Q63
  // m log2(e) as a 192-bit product p2:p1:p0 (log2(e) in Q127): value 2^(e - 1023), 190 fraction bits
  const uint64_t ch = 0xb8aa3b295c17f0bbull, cl = 0xbe87fed0691d3e89ull;
  const uint64_t p0 = m * cl, q = m * ch, r = umulhi(m, cl);
  const uint64_t p1 = q + r;
  const uint64_t p2 = umulhi(m, ch) + (p1 < q ? 1 : 0);
  // >> (190 - 124 - (e - 1023)) = 66 - (e - 1023), keeping 128 bits
  Wide o{0, 0};
  int s = 66 - (e - 1023);
  uint64_t a2 = p2, a1 = p1, a0 = p0;
  while (s >= 64) {
    a0 = a1;
    a1 = a2;
    a2 = 0;
    s -= 64;
    if (!a0 && !a1) return o;
  }
  if (s < 0) {   // |t| >= 2^67: the 64-bit sums wrap to nothing, the FP32 sum decides
    return o;
  }
  if (s) {
    a0 = (a0 >> s) | (a1 << (64 - s));
    a1 = (a1 >> s) | (a2 << (64 - s));
  }
  if (bt >> 63) {
    a0 = 0 - a0;
    a1 = ~a1 + (a0 == 0 ? 1 : 0);
  }
  o.hi = a1;
  o.lo = a0;
  return o;
}
// The Q60 part of k w for an integer k.
HPT_FX uint64_t times(int64_t k, const Wide& w) {
  return (uint64_t)k * w.hi + umulhi((uint64_t)k, w.lo) - (k < 0 ? w.lo : 0);
}

// An exponent sum: W modulo 16 (Q60) and the phase (Q64), which wrap around
// (unsigned: in signed arithmetic that would be undefined), and W in FP32.
struct Sum {
  uint64_t w, turn;
  float f;
};
// += a log y, for y's logarithm (l, turn, lf).
HPT_FX void add_power(Sum& s, int32_t a, uint64_t l, uint64_t turn, float lf) {
  s.w += (uint64_t)(int64_t)a * l;
  s.turn += (uint64_t)(int64_t)a * turn;
  s.f = fmaf((float)a, lf, s.f);
}

// cos and sin of theta (revolutions, Q64), Q62.  The nearest multiple of
// 1/4096 revolution comes from the tables, so multiples of a quarter turn give
// exactly 0 and +-1: what is real stays real.
HPT_FX void cossin(uint64_t th, const int64_t (*cs1)[2], const int64_t (*cs2)[2], int64_t& c, int64_t& s) {
  th += (uint64_t)1 << 51;
  const int i = (int)(th >> 58), j = (int)(th >> 52) & 63;
  const int64_t r = (int64_t)(th & (((uint64_t)1 << 52) - 1)) - ((int64_t)1 << 51);
  const int64_t c1 = cs1[i][0], s1 = cs1[i][1], c2 = cs2[j][0], s2 = cs2[j][1];
  const int64_t cc = mul62(c1, c2) - mul62(s1, s2), ss = mul62(s1, c2) + mul62(c1, s2);
  const int64_t f = mul62((int64_t)((uint64_t)r << 10), 0x3243f6a8885a308dll);   // phi = 2 pi r, Q71
  const int64_t p = mul62(f, f);                                                 // phi^2, Q80
  const int32_t ph = (int32_t)(p >> 32);                                         // Q48
  // kappa = 1 - cos phi = phi^2/2 - phi^4/24, Q62; sigma = sin phi = phi - phi^3/6, Q71
  const int64_t kap = (p >> 19) - mulhi32((int32_t)(((int64_t)ph * ph) >> 34), 178956971);
  const int64_t p6 = (int64_t)(((uint64_t)(p >> 28) * 715827883u) >> 32);         // phi^2/6, Q52
  const int64_t sg = f - (((int64_t)(int32_t)(f >> 32) * (int32_t)p6) >> 20);
  c = cc - mul62(cc, kap) - (mul62(ss, sg) >> 9);
  s = ss - mul62(ss, kap) + (mul62(cc, sg) >> 9);
}
// 2^f for the fraction f of W (Q60, its low 60 bits), in [1, 2), Q62.
HPT_FX int64_t exp2_frac(int64_t W, const int64_t* exp1, const int64_t* exp2) {
  const uint64_t f = (uint64_t)W << 4;
  const int64_t g64 = (int64_t)(f & (((uint64_t)1 << 52) - 1)) - ((int64_t)1 << 51);
  const int64_t e = mul62(exp1[f >> 58], exp2[(f >> 52) & 63]);
  const int64_t g = mul62((int64_t)((uint64_t)g64 << 10), 0x2c5c85fdf473de6bll);   // g ln 2, Q74
  const int32_t gh = (int32_t)(g >> 32);                                           // Q42
  // e^g - 1 = g + g (g/2 + g^2/6)
  const int32_t g2 = (int32_t)(((int64_t)gh * gh) >> 26);                          // g^2, Q58
  const int64_t s = (g >> 13) + (((int64_t)g2 * 715827883) >> 28);                 // Q62
  const int64_t h = g + mul62(g, s);
  return e + (mul62(e, h) >> 12);
}
// v 2^(k - 62) rounded to double, for results in the normal range (or v = 0).
HPT_FX double to_double(int64_t v, int k) {
  const uint64_t neg = (uint64_t)(v >> 63);
  uint64_t m = ((uint64_t)v ^ neg) - neg;
  const int lz = clz64(m | 1);
  m <<= lz;
  const uint64_t b = ((uint64_t)(k + 1023 - lz) << 52) + (((m >> 10) + 1) >> 1);   // the leading bit adds 1 to the exponent
  return of_bits(v == 0 ? 0 : b | (neg << 63));
}
// The same near and past the ends of the range: subnormal results, zero,
// infinity.
HPT_FX double to_double_any(int64_t v, int k) {
  if (k > 900) return to_double(v, k - 600) * 4.149515568880993e180;                         // 2^600
  if (k < -900) return k < -1200 ? 0.0 : to_double(v, k + 600) * 2.409919865102884e-181;     // 2^-600
  return to_double(v, k);
}

// The value of an exponent sum: 2^W (cos, sin)(2 pi turn), from the sum W
// modulo 16 (Q60), the phase and W in FP32 (within 7 of W).  exp_in: |wf| <=
// 900, no branches, so that a caller can interleave several; exp_of: every
// wf; past the range of a double 0, or NaN (over).
HPT_FX int exponent_of(int64_t W, float wf) {
  const int k4 = (int)(W >> 60);   // integer part modulo 16, in [-8, 8)
#ifdef __CUDA_ARCH__
  return k4 + 16 * __float2int_rn((wf - (float)k4) * 0.0625f);
#else
  return k4 + 16 * (int)lrintf((wf - (float)k4) * 0.0625f);
#endif
}
HPT_FX void exp_in(int64_t W, uint64_t turn, float wf, const int64_t* exp1, const int64_t* exp2,
                   const int64_t (*cs1)[2], const int64_t (*cs2)[2], double& er, double& ei) {
  int64_t c, s;
  cossin(turn, cs1, cs2, c, s);
  const int64_t m = exp2_frac(W, exp1, exp2);
  const int k = exponent_of(W, wf);
  er = to_double(mul62(m, c), k);
  ei = to_double(mul62(m, s), k);
}
HPT_FX bool exp_in_range(float wf) { return wf <= 900.f && wf >= -900.f; }
#ifdef __CUDACC__
__host__ __device__ __noinline__
#endif
static void exp_of(int64_t W, uint64_t turn, float wf, const int64_t* exp1, const int64_t* exp2,
                    const int64_t (*cs1)[2], const int64_t (*cs2)[2], double& er, double& ei) {
  if (!(wf < 1030.f)) {   // over the range, or a NaN in the sum
    er = ei = of_bits((uint64_t)0x7ff8 << 48);
    return;
  }
  if (wf < -1090.f) {
    er = ei = 0.0;
    return;
  }
  int64_t c, s;
  cossin(turn, cs1, cs2, c, s);
  const int64_t m = exp2_frac(W, exp1, exp2);
  const int k = exponent_of(W, wf);
  er = to_double_any(mul62(m, c), k);
  ei = to_double_any(mul62(m, s), k);
}

}  // namespace fx
}  // namespace hpt
