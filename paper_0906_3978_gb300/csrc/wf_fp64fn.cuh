// wf_fp64fn.cuh -- FP64 square root, quotient, logarithm and exponential in few FP64 operations.
//
// GB300 issues one FP64 operation per lane where the other pipes issue 64, so the FP64 steps of these
// functions are what they cost: ~10 for a division or square root, ~30 for a log or exp of the math library.
// Here the starting values come from FP32 reciprocal (square root) instructions, the logarithm and the
// exponential are table-driven (P.T.P. Tang, ACM TOMS 15 (1989) 144 and 16 (1990) 378): a short table
// brings the argument within 2^-7 (log) or 2^-7.5 (exp) of 1 or 0, where the Taylor series of degree 7 or 5
// reaches 2^-56.  All sign, exponent and index work is integer arithmetic.  Table values carry a second word, so
// that a function's error is its last rounding and little more: the window's values err no more than with the math
// library (rms over a 30-degree survey at 64^3 to 128^3: 2.27 to 2.59 units of 2^-53, as with the library;
// one-word tables 2.43 to 2.79).
#pragma once
#include "wf_common.cuh"
#include "wf_fntab.cuh"

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
// The rows come from memory (wf_fntab.cuh): making them with the math library's functions took each CTA 2 to 3 us
// of the FP64 pipe, more than the nodes of a small grid.
struct LogTable {
  double2 lg[kLogTab];  // (c, T = -log c)
};
struct FnTables {
  double c[kLogTab];
  double2 th[kLogTab];  // T as a multiple of 2^-40 and the rest
  double2 ex[kExpTab];  // 2^(j / 64) and what its rounding left
};
// fill the tables (in shared memory); a barrier has to follow
WF_D void load_log_table(LogTable& t, int tid, int nt) {
  for (int j = tid; j < kLogTab; j += nt) t.lg[j] = make_double2(kLogRows[j].c, kLogRows[j].th + kLogRows[j].tl);
}
WF_D void load_fn_tables(FnTables& t, int tid, int nt) {
  for (int j = tid; j < kLogTab; j += nt) {
    t.c[j] = kLogRows[j].c;
    t.th[j] = make_double2(kLogRows[j].th, kLogRows[j].tl);
  }
  for (int j = tid; j < kExpTab; j += nt) t.ex[j] = kExpRows[j];
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
// log(x), x positive and normal (13 FP64 operations): k log 2 + T as one exact sum of multiples of 2^-40, and the rest
WF_D double log_fast(double x, const FnTables& t) {
  const int hi = __double2hiint(x), ix = hi + (0x3ff00000 - 0x3fe80000);
  const int k = (ix >> 20) - 1023;
  const double m = __hiloint2double(hi - (k << 20), __double2loint(x));
  const int j = (ix >> 13) & (kLogTab - 1);
  const double2 th = t.th[j];
  const double kd = small_int(k), l = log1p_short(fma(m, t.c[j], -1.0));
  return fma(kd, 0x1.62e42fefa4p-1, th.x) + (l + fma(kd, -0x1.8432a1b0e2634p-43, th.y));  // log 2 in two parts
}
// exp(x) for -700 <= x <= 700 (12 FP64 operations)
WF_D double exp_fast(double x, const FnTables& tab) {
  const double s = fma(x, 92.33248261689366 /* 64 / log 2 */, 6755399441055744.0);  // 2^52 + 2^51 + n
  const int n = __double2loint(s);
  const double nd = s - 6755399441055744.0;
  // r = x - n log2 / 64, the constant in two parts (the first of 32 bits, so that n times it is exact)
  double r = fma(nd, -0x1.62e42feep-7, x);
  r = fma(nd, -0x1.a39ef35793c76p-39, r);
  double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
  p = fma(p, r, 1.0 / 6.0);
  p = fma(p, r, 0.5);
  const double2 t = tab.ex[n & (kExpTab - 1)];
  p = fma(p * r, r, r);
  return times_pow2(t.x + fma(t.x, p, t.y), n >> 6);
}

}  // namespace wf
