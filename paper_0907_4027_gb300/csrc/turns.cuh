// turns.cuh -- phases modulo one turn and their unit phasors, for the tables of the column and row
// phasors (tile_kernels.cuh).  Compiles as host code too (without FMA contraction): the test of its
// rounding runs there.
//
// A phase modulo one turn is a 64-bit fraction of a turn: a q and c q^2 (Eq. 2 per pixel index q) are
// integer products that drop whole turns by themselves, exact to 2^-64 |q| turns.  cos and sin of it:
// reduced to an eighth of a turn, Taylor series in the squared quarter turns, the leading three
// coefficients and their products in float-float (Dekker, Knuth), rounded once: within 0.501 ulp of the
// fraction's cos and sin, the correctly rounded value in all but 2 of 10^5 entries (with two coefficients
// in float-float, and the last 14 bits of the fraction dropped, 0.575 ulp and 0.08 % more rms error, in
// 26 instead of 35 us for 1920 x 1152 with 1000 traps; no difference that shows at 1024^2 with 256).
// No FP64 arithmetic: GB300 does ~2 FP64 operations per clock and SM, and FP64 sincospi made these
// tables 20 us of a 657 us frame at 512^2 with 100 traps and 230 us at 1920 x 1152 with 1000.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define HOT_TURNS_FN __device__ __forceinline__
#define HOT_TURNS_MUL(a, b) __fmul_rn(a, b)
#define HOT_TURNS_ADD(a, b) __fadd_rn(a, b)
#define HOT_TURNS_MULHI(a, b) __umul64hi(a, b)
#define HOT_TURNS_BITS(x) ((unsigned long long)__double_as_longlong(x))
#define HOT_TURNS_CLZ(x) __clzll((long long)(x))
#define HOT_TURNS_FLOAT(b) __uint_as_float(b)
#else
#include <math.h>
#include <string.h>
struct float2 {
  float x, y;
};
static inline float2 make_float2(float x, float y) {
  float2 v = {x, y};
  return v;
}
static inline unsigned long long hot_turns_bits(double x) {
  unsigned long long b;
  memcpy(&b, &x, 8);
  return b;
}
static inline float hot_turns_float(unsigned b) {
  float x;
  memcpy(&x, &b, 4);
  return x;
}
#define HOT_TURNS_FN static inline
#define HOT_TURNS_MUL(a, b) ((a) * (b))
#define HOT_TURNS_ADD(a, b) ((a) + (b))
#define HOT_TURNS_MULHI(a, b) ((unsigned long long)(((unsigned __int128)(a) * (b)) >> 64))
#define HOT_TURNS_BITS(x) hot_turns_bits(x)
#define HOT_TURNS_CLZ(x) __builtin_clzll(x)
#define HOT_TURNS_FLOAT(b) hot_turns_float(b)
#endif

namespace hot {

// |x| as a fixed-point number of fractions 2^-64, modulo 1 (truncated).
HOT_TURNS_FN unsigned long long turns_fixed(double x) {
  const unsigned long long b = HOT_TURNS_BITS(x);
  const int sh = (int)((b >> 52) & 0x7ff) - 1011;  // x = m 2^(sh - 64)
  const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
  return sh >= 64 || sh <= -64 ? 0ull : sh >= 0 ? m << sh : m >> -sh;
}

struct TrapTurns {
  unsigned long long a, c, cl;  // linear and quadratic turns per pixel index; cl: the next bits of |c|
  bool neg;                     // c < 0
};
HOT_TURNS_FN TrapTurns trap_turns(double lin, double quad) {
  TrapTurns t;
  t.a = turns_fixed(lin);
  if (lin < 0.0) t.a = 0ull - t.a;
  t.c = turns_fixed(quad);
  t.cl = turns_fixed(quad * 4294967296.0) << 32;  // (2^32: exact)
  t.neg = quad < 0.0;
  return t;
}
// a q + c q^2
HOT_TURNS_FN unsigned long long phase_at(const TrapTurns &k, int q) {
  const unsigned long long q2 = (unsigned long long)((long long)q * q);
  const unsigned long long t = k.c * q2 + HOT_TURNS_MULHI(k.cl, q2);
  return k.a * (unsigned long long)(long long)q + (k.neg ? 0ull - t : t);
}

// (h0 + l0) + (sh + sl) (bh + bl) in float-float, |h0| >= |sh bh|: the next Horner step.
HOT_TURNS_FN void horner_ff(float h0, float l0, float sh, float sl, float &bh, float &bl) {
  const float ph = HOT_TURNS_MUL(sh, bh), pl = fmaf(sh, bh, -ph) + fmaf(sh, bl, sl * bh);
  bh = HOT_TURNS_ADD(h0, ph);
  bl = HOT_TURNS_ADD(HOT_TURNS_ADD(h0, -bh), ph) + (pl + l0);
}

// cos and sin of a phase in fractions 2^-64 of a turn.
HOT_TURNS_FN float2 cis_turns(unsigned long long ph) {
  const unsigned n = (unsigned)((ph + (1ull << 61)) >> 62);  // quarter turns
  const long long r = (long long)(ph - ((unsigned long long)n << 62));
  // the rest in quarter turns, [-1/2, 1/2]: f + g, the leading 24 bits and the next 24 (by a shift: with
  // conversions of 64-bit integers a 1920 x 1152 trap set of 1000 took 38 us, this way 35)
  const unsigned long long a = r < 0 ? 0ull - (unsigned long long)r : (unsigned long long)r;
  const unsigned z = (unsigned)HOT_TURNS_CLZ(a | 1);
  const unsigned long long m = a << z;
  const unsigned sign = r < 0 ? 0x80000000u : 0u;
  const float f = (float)(int)(m >> 40) * HOT_TURNS_FLOAT(sign | ((105u - z) << 23));  // 2^(40 - 62 - z)
  const float g = (float)(int)((m >> 16) & 0xffffff) * HOT_TURNS_FLOAT(sign | ((81u - z) << 23));
  const float sh = HOT_TURNS_MUL(f, f), sl = fmaf(f, f, -sh) + 2.f * f * g;
  // sine: (f + g) (s0 + s (s1 + s (s2 + s p))), s_k = (-1)^k (pi/2)^(2k+1) / (2k+1)!
  float t = sh * fmaf(sh, fmaf(sh, -3.59884325e-06f, 1.60441181e-04f), -4.68175393e-03f);
  float vh = HOT_TURNS_ADD(0.0796926245f, t), vl = HOT_TURNS_ADD(HOT_TURNS_ADD(0.0796926245f, -vh), t) + 1.73683246e-09f;
  horner_ff(-0.645964086f, -1.14504903e-08f, sh, sl, vh, vl);
  horner_ff(1.57079637f, -4.37113883e-08f, sh, sl, vh, vl);
  const float sn = fmaf(f, vh, fmaf(f, vl, g * vh));
  // cosine: 1 + s (c1 + s (c2 + s p)), c_k = (-1)^k (pi/2)^(2k) / (2k)!
  t = sh * fmaf(sh, fmaf(sh, fmaf(sh, 4.71087475e-07f, -2.52020418e-05f), 9.19260259e-04f), -2.08634809e-02f);
  vh = HOT_TURNS_ADD(0.2536695f, t);
  vl = HOT_TURNS_ADD(HOT_TURNS_ADD(0.2536695f, -vh), t) + 7.55009566e-09f;
  horner_ff(-1.23370051f, -3.62964485e-08f, sh, sl, vh, vl);
  horner_ff(1.f, 0.f, sh, sl, vh, vl);
  const float co = vh + vl;
  const float x = n & 1 ? sn : co, y = n & 1 ? co : sn;
  return make_float2(n == 1 || n == 2 ? -x : x, n >= 2 ? -y : y);
}

}  // namespace hot
