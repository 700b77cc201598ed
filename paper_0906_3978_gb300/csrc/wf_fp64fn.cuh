// wf_fp64fn.cuh -- FP64 square root, quotient, logarithm and exponential in few FP64 operations.
//
// GB300 issues one FP64 operation per lane where the other pipes issue 64, so the FP64 steps of these
// functions are what they cost: ~10 for a division or square root, ~30 for a log or exp of the math library.
// Here the starting values come from FP32 reciprocal (square root) instructions, the logarithm and the
// exponential are table-driven (P.T.P. Tang, ACM TOMS 15 (1989) 144 and 16 (1990) 378): a short table
// brings the argument within 2^-7 (log) or 2^-7.5 (exp) of 1 or 0, where the Taylor series of degree 7 or 5
// reaches 2^-56.  All sign, exponent and index work is integer arithmetic.
#pragma once
#include "wf_common.cuh"

namespace wf {

// the double with a float's value (normal, positive) without a conversion on the FP64 pipe
WF_D double widen(float f) {
  const unsigned u = __float_as_uint(f);
  return __hiloint2double((int)((u >> 3) + (896u << 20)), (int)(u << 29));
}
// the leading bits of a positive normal double as a float times 2^-e; the value is f 2^e with f in [1, 2)
WF_D float lead(double d, int& e) {
  const int hi = __double2hiint(d);
  e = (hi >> 20) - 1023;
  return __uint_as_float(0x3f800000u | (((unsigned)hi << 3) & 0x7fffffu) | ((unsigned)__double2loint(d) >> 29));
}
// k as a double, without a conversion: 2^52 + 2^31 + k less 2^52 + 2^31
WF_D double small_int(int k) { return __hiloint2double(0x43300000, k ^ (int)0x80000000) - 4503601774854144.0; }
WF_D double times_pow2(double d, int e) { return __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d)); }

// sqrt(d) for a positive normal d (6 FP64 operations, within 1 ulp): Newton (Goldschmidt) from rsqrt in FP32
WF_D double sqrt_fast(double d) {
  int e;
  float f = lead(d, e);
  if (e & 1) f *= 2.f;  // d = f 4^h, f in [1, 4)
  const int h = (e - (e & 1)) / 2;
  const double x = times_pow2(d, -2 * h);
  const double y = widen(rsqrtf(f));
  double g = x * y, q = times_pow2(y, -1);
  const double s = fma(-g, q, 0.5);
  g = fma(g, s, g);
  q = fma(q, s, q);
  g = fma(fma(-g, g, x), q, g);
  return times_pow2(g, h);
}

// ---- logarithm -----------------------------------------------------------------------------------
// x = 2^k m with m in [3/4, 3/2); interval j of 128 gives c ~ 1/m and T = -log c (c = 1, T = 0 beside m = 1, so
// that log keeps its relative accuracy there); log x = k log 2 + T + log1p(m c - 1)
constexpr int kLogTab = 128, kExpTab = 64;
struct FnTables {
  double2 lg[kLogTab];  // (c, T); intervals of 1/256 from 3/4 to 1, of 1/128 from 1 to 3/2
  double ex[kExpTab];   // 2^(j / 64)
};
// fill the tables (in shared memory); a barrier has to follow
WF_D void make_fn_tables(FnTables& t, int tid, int nt) {
  for (int j = tid; j < kLogTab; j += nt) {
    const double mid = j < 64 ? 0.75 + (j + 0.5) / 256.0 : 1.0 + (j - 64 + 0.5) / 128.0;
    const double c = j == 63 || j == 64 ? 1.0 : rint(4096.0 / mid) / 4096.0;
    t.lg[j] = make_double2(c, c == 1.0 ? 0.0 : -log(c));
  }
  for (int j = tid; j < kExpTab; j += nt) t.ex[j] = exp2(j / 64.0);
}
// log1p(r) for |r| <= 2^-6.9
WF_D double log1p_short(double r) {
  double p = fma(r, 1.0 / 7.0, -1.0 / 6.0);
  p = fma(p, r, 0.2);
  p = fma(p, r, -0.25);
  p = fma(p, r, 1.0 / 3.0);
  p = fma(p, r, -0.5);
  return fma(p * r, r, r);
}
// log(x), x positive and normal (11 FP64 operations)
WF_D double log_fast(double x, const double2* __restrict__ lg) {
  const int hi = __double2hiint(x), ix = hi + (0x3ff00000 - 0x3fe80000);
  const int k = (ix >> 20) - 1023;
  const double m = __hiloint2double(hi - (k << 20), __double2loint(x));
  const double2 t = lg[(ix >> 13) & (kLogTab - 1)];
  const double r = fma(m, t.x, -1.0);
  return fma(small_int(k), 0.69314718055994530942, t.y + log1p_short(r));
}
// exp(x) for -700 <= x <= 700 (11 FP64 operations)
WF_D double exp_fast(double x, const double* __restrict__ ex) {
  const double s = fma(x, 92.33248261689366 /* 64 / log 2 */, 6755399441055744.0);  // 2^52 + 2^51 + n
  const int n = __double2loint(s);
  const double nd = s - 6755399441055744.0;
  // r = x - n log2 / 64, the constant in two parts (the first of 32 bits, so that n times it is exact)
  double r = fma(nd, -0x1.62e42feep-7, x);
  r = fma(nd, -0x1.a39ef35793c76p-39, r);
  double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
  p = fma(p, r, 1.0 / 6.0);
  p = fma(p, r, 0.5);
  const double t = ex[n & (kExpTab - 1)];
  p = fma(p * r, r, r);
  return times_pow2(fma(t, p, t), n >> 6);
}

}  // namespace wf
