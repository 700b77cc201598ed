// wf_fix.cuh -- transforms of FP64 data in 64-bit fixed point.
//
// GB300's FP64 pipe issues one operation per lane where the integer and FP32 pipes issue 64, so an
// FP64 butterfly is bound by that pipe alone (an 8-point butterfly with its seven twiddles: 50.6
// Gpoints/s over the chip in FP64).  The same butterfly on 64-bit integers, twiddles as Q62 digits,
// runs at 429 Gpoints/s: additions are two integer instructions and a complex product twelve 32 x 32
// -> 64 multiply-adds, about the time of one FP64 operation.
//
// A line of M complex values z is scaled by a power of two so that sqrt(M) ||z||_2 <= 2^62.  By
// Cauchy-Schwarz every partial sum of its DFT then stays below 2^62 in modulus, so no later step
// rescales, and one unit is at most 2^-62 sqrt(M) of the output's rms: with the one or two units
// of rounding noise a transform adds, ~1e-17 relative at M = 512, where FP64 butterflies leave ~2e-16.
// What remains is the rounding of the FP64 values that are stored.  A line's scale comes from its own
// largest exponent and sum of squares, so lines of any magnitude keep their digits; the statistics are
// integers, so the result does not depend on the order in which threads add to them.  A line with an
// infinity or NaN becomes NaN throughout (FP64 butterflies spread either over the line as well).
#pragma once
#include <type_traits>

#include "wf_line.cuh"

namespace wf {

struct fxc {
  long long x, y;
};
WF_D fxc operator+(fxc a, fxc b) { return fxc{a.x + b.x, a.y + b.y}; }
WF_D fxc operator-(fxc a, fxc b) { return fxc{a.x - b.x, a.y - b.y}; }
// a * i * DIR
template <int DIR> WF_D fxc fx_mul_i(fxc a) { return DIR > 0 ? fxc{-a.y, a.x} : fxc{a.y, -a.x}; }

WF_D long long fx_mad(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
WF_D long long fx_mul(int a, int b) {
  long long r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
// balanced digits: a = h 2^32 + l with l the signed low word
WF_D void fx_digits(long long a, int& h, int& l) {
  l = (int)a;
  h = (int)(a >> 32) - (l >> 31);
}
// a w for a Q62 factor w = wh 2^32 + wl (|w| <= 1), rounded to a unit (the product of the two low
// digits, below one unit, is left out).  |a| < 2^62.5
WF_D long long fx_mulq(long long a, int wh, int wl) {
  int h, l;
  fx_digits(a, h, l);
  return (fx_mul(h, wh) << 2) + (fx_mad(l, wh, fx_mad(h, wl, 1ll << 29)) >> 30);
}
// a w (DIR < 0) or a conj(w) (DIR > 0) for w = (w.x, w.y | w.z, w.w) digits of Q62 re and im, |w| <= 1 and
// |a| <= 2^62: the high products stay below 2^60 and the middle sums below 2^62.6
// (w's digits are negated, never a's: a low digit of a may be -2^31, those of the tables are not)
template <int DIR> WF_D fxc fx_twid(fxc a, int4 w) {
  int hr, lr, hi, li;
  fx_digits(a.x, hr, lr);
  fx_digits(a.y, hi, li);
  // (zx, wx): the digits that multiply a.y in the real part, (zy, wy): a.x in the imaginary part
  const int zx = DIR < 0 ? -w.z : w.z, wx = DIR < 0 ? -w.w : w.w;
  const int zy = DIR < 0 ? w.z : -w.z, wy = DIR < 0 ? w.w : -w.w;
  const long long hx = fx_mad(hi, zx, fx_mul(hr, w.x));
  const long long mx = fx_mad(li, zx, fx_mad(hi, wx, fx_mad(lr, w.x, fx_mad(hr, w.y, 1ll << 29))));
  const long long hy = fx_mad(hi, w.x, fx_mul(hr, zy));
  const long long my = fx_mad(li, w.x, fx_mad(hi, w.y, fx_mad(lr, zy, fx_mad(hr, wy, 1ll << 29))));
  return fxc{(hx << 2) + (mx >> 30), (hy << 2) + (my >> 30)};
}
// Q62 digits of cos and sin of the constant rotations
constexpr int kFxR2h = 759250125, kFxR2l = -25716447;       // sqrt(1/2)
constexpr int kFxS3h = 929887697, kFxS3l = -1332128537;     // sqrt(3)/2
// exp(-2 pi i m / 9), m = 1, 2, 4
WF_D int4 fx_w9(int m) {
  return m == 1 ? make_int4(822533958, -1633652124, -690187940, -2016164183)
         : m == 2 ? make_int4(186453311, 96060625, -1057429273, -37236404)
                  : make_int4(-1008987269, 1537591498, -367241333, 1978927779);
}

// ---- radix plans: M = R1 R2 R3 (R3 = 1: two passes), butterflies of up to 12 points ------
struct FxRad {
  int r1, r2, r3;
};
// (the last radix no smaller than the first, or a divisor of it, so that no pass runs a nearly empty round)
constexpr FxRad fx_plan(int m) {
  switch (m) {
    case 8: return {4, 2, 1};
    case 12: return {3, 4, 1};
    case 16: return {4, 4, 1};
    case 24: return {4, 6, 1};
    case 32: return {8, 4, 1};
    case 36: return {6, 6, 1};
    case 48: return {6, 8, 1};
    case 54: return {6, 9, 1};
    case 64: return {8, 8, 1};
    case 72: return {8, 9, 1};
    case 96: return {8, 12, 1};
    case 108: return {9, 12, 1};
    case 128: return {8, 4, 4};
    case 144: return {12, 12, 1};
    case 192: return {8, 6, 4};
    case 216: return {6, 6, 6};
    case 256: return {8, 8, 4};
    case 288: return {6, 6, 8};
    case 384: return {6, 8, 8};
    case 512: return {8, 8, 8};
    default: return {0, 0, 0};
  }
}

// the operations of the line engine (wf_line.cuh) on fixed-point values
template <int DIR> WF_D fxc ln_mul_i(fxc a) { return fx_mul_i<DIR>(a); }
template <int DIR> WF_D fxc ln_twid(fxc a, int4 w) { return fx_twid<DIR>(a, w); }
WF_D fxc ln_r2(fxc a) { return fxc{fx_mulq(a.x, kFxR2h, kFxR2l), fx_mulq(a.y, kFxR2h, kFxR2l)}; }
WF_D fxc ln_s3(fxc a) { return fxc{fx_mulq(a.x, kFxS3h, kFxS3l), fx_mulq(a.y, kFxS3h, kFxS3l)}; }
WF_D fxc ln_half(fxc a) { return fxc{(a.x + 1) >> 1, (a.y + 1) >> 1}; }
template <int DIR> WF_D fxc ln_rot9(fxc a, int m) { return fx_twid<DIR>(a, fx_w9(m)); }

// radix plan of a fixed-point line: butterflies of at most 12 points
template <int M> struct FxPlan {
  static constexpr int r1 = fx_plan(M).r1, r2 = fx_plan(M).r2, r3 = fx_plan(M).r3;
};

// ---- scaling -----------------------------------------------------------------------------------
WF_D int fx_exp(double d) { return (__double2hiint(d) >> 20) & 0x7ff; }
// an upper bound of |d| 2^(12 - (emax - 1023)), 13 bits and one, for exponents up to emax (where SUB is false, a
// subnormal's is 1: emax is at least 14)
template <bool SUB = false> WF_D unsigned fx_top(double d, int emax) {
  const int hi = __double2hiint(d), e = (hi >> 20) & 0x7ff;
  if constexpr (SUB) {
    const int s = emax - max(e, 1) + 8;
    const unsigned m = (unsigned)(hi & 0xfffff) | (e ? 0x100000u : 0u);
    return s > 31 || m == 0 ? (unsigned)((m | (unsigned)__double2loint(d)) != 0) : (m >> s) + 1u;
  }
  const int s = emax - e + 8;
  return e == 0 || s > 31 ? (unsigned)((hi & 0x7fffffff) != 0 || __double2loint(d) != 0)
                          : ((unsigned)((hi & 0xfffff) | 0x100000) >> s) + 1u;
}
// 2^e for -1022 <= e <= 1023
WF_D double fx_pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }
// d 2^e for any e; the result under- or overflows as it should
WF_D double fx_scaled(double d, int e) {
  e = min(max(e, -2044), 2044);
  return d * fx_pow2(e / 2) * fx_pow2(e - e / 2);
}
// d 2^k rounded to an integer (0 where the exponent leaves the normal range downwards)
WF_D long long fx_from(double d, int k) {
  const int hi = __double2hiint(d), e = (hi >> 20) & 0x7ff;
  if (e == 0 || e + k <= 0) return 0;
  return __double2ll_rn(__hiloint2double(hi + (k << 20), __double2loint(d)));
}
// The power of two k that takes a line of M complex values to sqrt(M) ||z||_2 2^k <= 2^62: emax the
// largest biased exponent of the line, q >= (sum of fx_top^2) / 128
WF_D int fx_scale(int emax, unsigned q, int M) {
  const unsigned long long s = (unsigned long long)q * 128ull * (unsigned)M;
  const int b = 64 - __clzll((long long)s);  // sqrt(s) < 2^(b / 2)
  return 62 - (emax - 1023) + 12 - ((b + 1) >> 1);
}

// A line's scale: its values are integers in units of 2^-k; nan: the exponent bits that make every
// result of a line with a non-finite element a NaN.  kMin: the smallest exponent a line is taken to have: 2^-800,
// below which values keep the resolution of 2^-860.
struct FxScale {
  static constexpr int kMin = 223;
  int k;
  unsigned nan;
};
// The same for the whole FP64 range, in the passes of a filter on a caller's field and of a residual: integers are made
// from the registers' values by 2^kin, and scalings past 2^+-kFxStep, which an exponent field may not hold, are
// multiplications.  (In the passes of a CG iteration, whose smallest values are sqrt(the smallest norm), it
// costs 3 to 5% of an FP64 solve and can change nothing.)
constexpr int kFxStep = 900;
struct FxWide {
  static constexpr int kMin = 1;
  int k, kin;
  unsigned nan;
};
// The scale of the line whose elements are spread over the threads' raw[]; se, sq: the line's words in
// shared memory, S::kMin and 0 before (visible to all).  Two barriers.  In the wide form a line of zeros gets k = 0,
// and the values of a line of tiny ones, subnormals among them, are multiplied by 2^600 in the registers.
template <class S = FxScale, int NV> WF_D S fx_line_scale(double2 (&raw)[NV], int* se, unsigned* sq, int M) {
  static_assert(2 * NV <= 62, "the sum of squares of a thread fits 32 bits");
  constexpr bool WIDE = std::is_same<S, FxWide>::value;
  int mx = 0;
#pragma unroll
  for (int r = 0; r < NV; ++r) mx = max(mx, max(fx_exp(raw[r].x), fx_exp(raw[r].y)));
  if (mx > S::kMin) atomicMax(se, mx);
  __syncthreads();
  const int emax = *se;
  unsigned q = 0;
#pragma unroll
  for (int r = 0; r < NV; ++r) {
    const unsigned h0 = fx_top<WIDE>(raw[r].x, emax), h1 = fx_top<WIDE>(raw[r].y, emax);
    q += h0 * h0 + h1 * h1;
  }
  if (q) atomicAdd(sq, (q >> 7) + 1u);
  __syncthreads();
  const unsigned nan = emax == 0x7ff ? 0x7ff80000u : 0u;
  if constexpr (WIDE) {
    const unsigned s = *sq;
    FxWide f{s ? fx_scale(emax, s + 1u, M) : 0, 0, nan};
    f.kin = f.k;
    if (f.k > kFxStep) {
      f.kin = f.k - 600;
#pragma unroll
      for (int r = 0; r < NV; ++r) raw[r] = make_double2(raw[r].x * 0x1p600, raw[r].y * 0x1p600);
    }
    return f;
  } else {
    return FxScale{fx_scale(emax, *sq + 1u, M), nan};
  }
}
WF_D fxc fx_from2(double2 d, FxScale f) { return fxc{fx_from(d.x, f.k), fx_from(d.y, f.k)}; }
WF_D fxc fx_from2(double2 d, FxWide f) { return fxc{fx_from(d.x, f.kin), fx_from(d.y, f.kin)}; }
// v 2^-(k + sh).  The power of two goes to the exponent field by an integer addition (values near the top
// of the range, where it could overflow, take a multiplication).
template <class S> WF_D double fx_to(long long v, S f, int sh = 0) {
  const int k = f.k + sh;
  double d = __ll2double_rn(v);
  if constexpr (std::is_same<S, FxWide>::value) {
    if ((unsigned)(k + kFxStep) > 2u * kFxStep) d = fx_scaled(d, -k);
    else if (v != 0) d = __hiloint2double(__double2hiint(d) - (k << 20), __double2loint(d));
  } else {
    if (k < -900) d *= fx_pow2(-k);
    else if (v != 0) d = __hiloint2double(__double2hiint(d) - (k << 20), __double2loint(d));
  }
  return __hiloint2double(__double2hiint(d) | (int)f.nan, __double2loint(d));
}
template <class S> WF_D double2 fx_to2(fxc v, S f, int sh = 0) { return make_double2(fx_to(v.x, f, sh), fx_to(v.y, f, sh)); }
WF_D long long fx_rshift(long long v, int s) { return (v + (1ll << (s - 1))) >> s; }  // s >= 1, rounded

constexpr int fx_floor_log2(int n) { return n < 2 ? 0 : 1 + fx_floor_log2(n / 2); }
// the shift between a forward transform and the inverse that follows: ceil(log2(n) / 2), since the inverse's
// partial sums are below n ||z||_2, sqrt(n) times the forward's
constexpr int fx_mid(int n) { return (fx_floor_log2(n - 1) + 2) / 2; }

// twiddles exp(-2 pi i e / N), e < N, of the table exp(-2 pi i e / 2N) in shared memory
template <int N> WF_D void fx_load_tw(int4* tw, const int4* __restrict__ tab, int tid, int nt) {
  for (int e = tid; e < N; e += nt) tw[e] = __ldg(tab + 2 * e);
}

}  // namespace wf
