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
// integers, so the result does not depend on the order in which threads add to them.  Lines whose
// largest value lies below 2^-800 keep an absolute resolution of about 2^-860 only, and a line with an
// infinity or NaN becomes NaN throughout (FP64 butterflies spread either over the line as well).
#pragma once
#include "wf_common.cuh"

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

// ---- small DFTs in registers ---------------------------------------------------------------
template <int DIR> WF_D void fx_dft2(fxc& a, fxc& b) {
  const fxc s = a + b;
  b = a - b;
  a = s;
}
template <int DIR> WF_D void fx_dft3(fxc& a, fxc& b, fxc& c) {
  const fxc t = b + c, u = b - c;
  const fxc m{a.x - ((t.x + 1) >> 1), a.y - ((t.y + 1) >> 1)};
  const fxc ju = fx_mul_i<DIR>(fxc{fx_mulq(u.x, kFxS3h, kFxS3l), fx_mulq(u.y, kFxS3h, kFxS3l)});
  a = a + t;
  b = m + ju;
  c = m - ju;
}
template <int DIR> WF_D void fx_dft4(fxc& a, fxc& b, fxc& c, fxc& d) {
  const fxc t0 = a + c, t1 = a - c, t2 = b + d, t3 = fx_mul_i<DIR>(b - d);
  a = t0 + t2;
  b = t1 + t3;
  c = t0 - t2;
  d = t1 - t3;
}
// v[0..RAD) -> its DFT in natural order
template <int RAD, int DIR> WF_D void fx_dft(fxc* v) {
  if constexpr (RAD == 2) {
    fx_dft2<DIR>(v[0], v[1]);
  } else if constexpr (RAD == 3) {
    fx_dft3<DIR>(v[0], v[1], v[2]);
  } else if constexpr (RAD == 4) {
    fx_dft4<DIR>(v[0], v[1], v[2], v[3]);
  } else if constexpr (RAD == 6) {
    // 2 x 3 without twiddles: n = 3 n1 + 2 n2, k = 3 k1 + 4 k2 (mod 6)
    fxc a0 = v[0], a1 = v[2], a2 = v[4], b0 = v[3], b1 = v[5], b2 = v[1];
    fx_dft3<DIR>(a0, a1, a2);
    fx_dft3<DIR>(b0, b1, b2);
    v[0] = a0 + b0;
    v[3] = a0 - b0;
    v[4] = a1 + b1;
    v[1] = a1 - b1;
    v[2] = a2 + b2;
    v[5] = a2 - b2;
  } else if constexpr (RAD == 8) {
    fx_dft4<DIR>(v[0], v[2], v[4], v[6]);
    fx_dft4<DIR>(v[1], v[3], v[5], v[7]);
    // W8^1 = (1 + DIR i)/sqrt2, W8^2 = DIR i, W8^3 = (-1 + DIR i)/sqrt2
    const fxc p = v[3] + fx_mul_i<DIR>(v[3]), q = fx_mul_i<DIR>(v[7]) - v[7];
    const fxc o1{fx_mulq(p.x, kFxR2h, kFxR2l), fx_mulq(p.y, kFxR2h, kFxR2l)};
    const fxc o2 = fx_mul_i<DIR>(v[5]);
    const fxc o3{fx_mulq(q.x, kFxR2h, kFxR2l), fx_mulq(q.y, kFxR2h, kFxR2l)};
    const fxc e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
    v[0] = e0 + o0;
    v[4] = e0 - o0;
    v[1] = e1 + o1;
    v[5] = e1 - o1;
    v[2] = e2 + o2;
    v[6] = e2 - o2;
    v[3] = e3 + o3;
    v[7] = e3 - o3;
  } else if constexpr (RAD == 9) {
    // 3 x 3: columns n = 3 n1 + n2, twiddles W9^(n2 k1), rows; k = k1 + 3 k2
    fx_dft3<DIR>(v[0], v[3], v[6]);
    fx_dft3<DIR>(v[1], v[4], v[7]);
    fx_dft3<DIR>(v[2], v[5], v[8]);
    v[4] = fx_twid<DIR>(v[4], fx_w9(1));
    v[5] = fx_twid<DIR>(v[5], fx_w9(2));
    v[7] = fx_twid<DIR>(v[7], fx_w9(2));
    v[8] = fx_twid<DIR>(v[8], fx_w9(4));
    fx_dft3<DIR>(v[0], v[1], v[2]);
    fx_dft3<DIR>(v[3], v[4], v[5]);
    fx_dft3<DIR>(v[6], v[7], v[8]);
    fxc t = v[1];  // transpose the 3 x 3 result
    v[1] = v[3];
    v[3] = t;
    t = v[2];
    v[2] = v[6];
    v[6] = t;
    t = v[5];
    v[5] = v[7];
    v[7] = t;
  } else {
    static_assert(RAD == 12, "radix");
    // 4 x 3 without twiddles: n = 3 n1 + 4 n2, k = 9 k1 + 4 k2 (mod 12)
    fxc a[3][4];
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < 4; ++n1) a[n2][n1] = v[(3 * n1 + 4 * n2) % 12];
      fx_dft4<DIR>(a[n2][0], a[n2][1], a[n2][2], a[n2][3]);
    }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      fx_dft3<DIR>(a[0][k1], a[1][k1], a[2][k1]);
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) v[(9 * k1 + 4 * k2) % 12] = a[k2][k1];
    }
  }
}

// ---- radix plans: M = R1 R2 R3 (R3 = 1: two passes), butterflies small enough for registers ------
struct FxRad {
  int r1, r2, r3;
};
constexpr FxRad fx_plan(int m) {
  switch (m) {
    case 8: return {4, 2, 1};
    case 12: return {4, 3, 1};
    case 16: return {4, 4, 1};
    case 24: return {6, 4, 1};
    case 32: return {8, 4, 1};
    case 36: return {6, 6, 1};
    case 48: return {8, 6, 1};
    case 54: return {9, 6, 1};
    case 64: return {8, 8, 1};
    case 72: return {12, 6, 1};
    case 96: return {12, 8, 1};
    case 108: return {12, 9, 1};
    case 128: return {8, 4, 4};
    case 144: return {12, 12, 1};
    case 192: return {8, 6, 4};
    case 216: return {6, 6, 6};
    case 256: return {8, 8, 4};
    case 288: return {8, 6, 6};
    case 384: return {8, 8, 6};
    case 512: return {8, 8, 8};
    default: return {0, 0, 0};
  }
}

// Forward transform, a multiplier at each k, and the inverse transform (unnormalised) of one line held
// by TPL = M / R1 threads: thread t enters with v[n1] = z[n1 (M / R1) + t] and leaves with the same
// elements of the result.  n = n1 R2 R3 + n2 R3 + n3, k = k1 + R1 k2 + R1 R2 k3; every pass writes the
// slots it read, so one barrier stands between two passes.  s: the line's M slots (slot p at
// s[map(p)]); tw[e] = digits of exp(-2 pi i e / M); ph(k, X): the multiplier.  Every thread of the CTA
// calls it; all of the CTA's lines are done together.
template <int M, class MAP, class PH>
WF_D void fx_convolve(fxc (&v)[fx_plan(M).r1], fxc* s, const MAP& map, int t, const int4* tw, const PH& ph) {
  constexpr int R1 = fx_plan(M).r1, R2 = fx_plan(M).r2, R3 = fx_plan(M).r3, N1 = M / R1;
  static_assert(R1 * R2 * R3 == M, "plan");
  fx_dft<R1, -1>(v);
  s[map(t)] = v[0];
#pragma unroll
  for (int k1 = 1; k1 < R1; ++k1) s[map(k1 * N1 + t)] = fx_twid<-1>(v[k1], tw[t * k1]);
  __syncthreads();
  if constexpr (R3 > 1) {
    for (int j = t; j < M / R2; j += N1) {
      const int k1 = j / R3, n3 = j % R3, base = k1 * R2 * R3 + n3;
      fxc a[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) a[n2] = s[map(base + n2 * R3)];
      fx_dft<R2, -1>(a);
      s[map(base)] = a[0];
#pragma unroll
      for (int k2 = 1; k2 < R2; ++k2) s[map(base + k2 * R3)] = fx_twid<-1>(a[k2], tw[R1 * n3 * k2]);
    }
    __syncthreads();
    for (int j = t; j < M / R3; j += N1) {
      const int k1 = j / R2, k2 = j % R2, base = j * R3;
      fxc a[R3];
#pragma unroll
      for (int n3 = 0; n3 < R3; ++n3) a[n3] = s[map(base + n3)];
      fx_dft<R3, -1>(a);
#pragma unroll
      for (int k3 = 0; k3 < R3; ++k3) a[k3] = ph(k1 + R1 * k2 + R1 * R2 * k3, a[k3]);
      fx_dft<R3, +1>(a);
      s[map(base)] = a[0];
#pragma unroll
      for (int n3 = 1; n3 < R3; ++n3) s[map(base + n3)] = fx_twid<+1>(a[n3], tw[R1 * n3 * k2]);
    }
    __syncthreads();
    for (int j = t; j < M / R2; j += N1) {
      const int k1 = j / R3, n3 = j % R3, base = k1 * R2 * R3 + n3;
      fxc a[R2];
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) a[k2] = s[map(base + k2 * R3)];
      fx_dft<R2, +1>(a);
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) s[map(base + n2 * R3)] = fx_twid<+1>(a[n2], tw[(n2 * R3 + n3) * k1]);
    }
  } else {
    for (int j = t; j < R1; j += N1) {  // j = k1
      fxc a[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) a[n2] = s[map(j * R2 + n2)];
      fx_dft<R2, -1>(a);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) a[k2] = ph(j + R1 * k2, a[k2]);
      fx_dft<R2, +1>(a);
      s[map(j * R2)] = a[0];
#pragma unroll
      for (int n2 = 1; n2 < R2; ++n2) s[map(j * R2 + n2)] = fx_twid<+1>(a[n2], tw[n2 * j]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) v[k1] = s[map(k1 * N1 + t)];
  fx_dft<R1, +1>(v);
}

// The forward half alone, in either direction (DIR = +1: conjugate twiddles): enters like fx_convolve
// and hands every Z_k the thread ends with to out(k, Z_k, i), i = 0, 1, ... its number in the thread.  TWS: W_M^e = tw[TWS e].
template <int M, int DIR, int TWS = 1, class MAP, class OUT>
WF_D void fx_forward(fxc (&v)[fx_plan(M).r1], fxc* s, const MAP& map, int t, const int4* tw, const OUT& out) {
  constexpr int R1 = fx_plan(M).r1, R2 = fx_plan(M).r2, R3 = fx_plan(M).r3, N1 = M / R1;
  fx_dft<R1, DIR>(v);
  s[map(t)] = v[0];
#pragma unroll
  for (int k1 = 1; k1 < R1; ++k1) s[map(k1 * N1 + t)] = fx_twid<DIR>(v[k1], tw[TWS * t * k1]);
  __syncthreads();
  if constexpr (R3 > 1) {
    for (int j = t; j < M / R2; j += N1) {
      const int k1 = j / R3, n3 = j % R3, base = k1 * R2 * R3 + n3;
      fxc a[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) a[n2] = s[map(base + n2 * R3)];
      fx_dft<R2, DIR>(a);
      s[map(base)] = a[0];
#pragma unroll
      for (int k2 = 1; k2 < R2; ++k2) s[map(base + k2 * R3)] = fx_twid<DIR>(a[k2], tw[TWS * R1 * n3 * k2]);
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < (M / R3 + N1 - 1) / N1; ++m) {
      const int j = t + m * N1;
      if ((M / R3) % N1 == 0 || j < M / R3) {
        fxc a[R3];
#pragma unroll
        for (int n3 = 0; n3 < R3; ++n3) a[n3] = s[map(j * R3 + n3)];
        fx_dft<R3, DIR>(a);
#pragma unroll
        for (int k3 = 0; k3 < R3; ++k3) out(j / R2 + R1 * (j % R2) + R1 * R2 * k3, a[k3], m * R3 + k3);
      }
    }
  } else {
#pragma unroll
    for (int m = 0; m < (R1 + N1 - 1) / N1; ++m) {
      const int j = t + m * N1;
      if (R1 % N1 == 0 || j < R1) {
        fxc a[R2];
#pragma unroll
        for (int n2 = 0; n2 < R2; ++n2) a[n2] = s[map(j * R2 + n2)];
        fx_dft<R2, DIR>(a);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) out(j + R1 * k2, a[k2], m * R2 + k2);
      }
    }
  }
}

// The same with the result left in the line's slots in natural order (a barrier after it).
template <int M, int DIR, int TWS, class MAP>
WF_D void fx_forward_nat(fxc (&v)[fx_plan(M).r1], fxc* s, const MAP& map, int t, const int4* tw) {
  constexpr int R1 = fx_plan(M).r1, R2 = fx_plan(M).r2, R3 = fx_plan(M).r3, N1 = M / R1;
  constexpr int RL = R3 > 1 ? R3 : R2, NB = M / RL, PER = (NB + N1 - 1) / N1;
  fxc res[PER * RL];
  fx_forward<M, DIR, TWS>(v, s, map, t, tw, [&](int, fxc X, int i) { res[i] = X; });
  __syncthreads();
#pragma unroll
  for (int m = 0; m < PER; ++m) {
    const int j = t + m * N1;
    if (NB % N1 == 0 || j < NB)
#pragma unroll
      for (int r = 0; r < RL; ++r) s[map(R3 > 1 ? j / R2 + R1 * (j % R2) + R1 * R2 * r : j + R1 * r)] = res[m * RL + r];
  }
  __syncthreads();
}

// The mirror image: takes Z_k from in(k) (which may read the line's own slots: a barrier stands before
// the first write) and leaves v[n1] = z[n1 (M / R1) + t], z_n = sum_k Z_k exp(DIR 2 pi i k n / M).
template <int M, int DIR, int TWS = 1, class MAP, class IN>
WF_D void fx_inverse(fxc (&v)[fx_plan(M).r1], fxc* s, const MAP& map, int t, const int4* tw, const IN& in) {
  constexpr int R1 = fx_plan(M).r1, R2 = fx_plan(M).r2, R3 = fx_plan(M).r3, N1 = M / R1;
  constexpr int RL = R3 > 1 ? R3 : R2, NB = M / RL, PER = (NB + N1 - 1) / N1;
  fxc a[PER][RL];
#pragma unroll
  for (int m = 0; m < PER; ++m) {
    const int j = t + m * N1;
    if (NB % N1 == 0 || j < NB)
#pragma unroll
      for (int r = 0; r < RL; ++r)
        a[m][r] = R3 > 1 ? in(j / R2 + R1 * (j % R2) + R1 * R2 * r) : in(j + R1 * r);
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < PER; ++m) {
    const int j = t + m * N1;
    if (NB % N1 == 0 || j < NB) {
      fx_dft<RL, DIR>(a[m]);
      const int e = R3 > 1 ? R1 * (j % R2) : j;  // twiddle step of output r
      s[map(j * RL)] = a[m][0];
#pragma unroll
      for (int r = 1; r < RL; ++r) s[map(j * RL + r)] = fx_twid<DIR>(a[m][r], tw[TWS * r * e]);
    }
  }
  __syncthreads();
  if constexpr (R3 > 1) {
    for (int j = t; j < M / R2; j += N1) {
      const int k1 = j / R3, n3 = j % R3, base = k1 * R2 * R3 + n3;
      fxc b[R2];
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) b[k2] = s[map(base + k2 * R3)];
      fx_dft<R2, DIR>(b);
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) s[map(base + n2 * R3)] = fx_twid<DIR>(b[n2], tw[TWS * (n2 * R3 + n3) * k1]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) v[k1] = s[map(k1 * N1 + t)];
  fx_dft<R1, DIR>(v);
}

// ---- scaling -----------------------------------------------------------------------------------
WF_D int fx_exp(double d) { return (__double2hiint(d) >> 20) & 0x7ff; }
// an upper bound of |d| 2^(12 - (emax - 1023)), 13 bits and one, for exponents up to emax
WF_D unsigned fx_top(double d, int emax) {
  const int hi = __double2hiint(d), e = (hi >> 20) & 0x7ff, s = emax - e + 8;
  return e == 0 || s > 31 ? (unsigned)((hi & 0x7fffffff) != 0 || __double2loint(d) != 0)
                          : ((unsigned)((hi & 0xfffff) | 0x100000) >> s) + 1u;
}
// d 2^k rounded to an integer (0 where the exponent leaves the normal range downwards)
WF_D long long fx_from(double d, int k) {
  const int hi = __double2hiint(d), e = (hi >> 20) & 0x7ff;
  if (e == 0 || e + k <= 0) return 0;
  return __double2ll_rn(__hiloint2double(hi + (k << 20), __double2loint(d)));
}
// 2^e for -1022 <= e <= 1023
WF_D double fx_pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }
// The power of two k that takes a line of M complex values to sqrt(M) ||z||_2 2^k <= 2^62: emax the
// largest biased exponent of the line (at least kFxMinExp), q >= (sum of fx_top^2) / 128
constexpr int kFxMinExp = 223;
WF_D int fx_scale(int emax, unsigned q, int M) {
  const unsigned long long s = (unsigned long long)q * 128ull * (unsigned)M;
  const int b = 64 - __clzll((long long)s);  // sqrt(s) < 2^(b / 2)
  return 62 - (emax - 1023) + 12 - ((b + 1) >> 1);
}


// A line's scale: its values are integers in units of 2^-k; nan: the exponent bits that make every
// result of a line with a non-finite element a NaN
struct FxScale {
  int k;
  unsigned nan;
};
// The scale of the line whose elements are spread over the threads' raw[]; se, sq: the line's words in
// shared memory, kFxMinExp and 0 before (visible to all).  Two barriers.
template <int NV> WF_D FxScale fx_line_scale(const double2 (&raw)[NV], int* se, unsigned* sq, int M) {
  static_assert(2 * NV <= 62, "the sum of squares of a thread fits 32 bits");
  int mx = 0;
#pragma unroll
  for (int r = 0; r < NV; ++r) mx = max(mx, max(fx_exp(raw[r].x), fx_exp(raw[r].y)));
  if (mx > kFxMinExp) atomicMax(se, mx);
  __syncthreads();
  const int emax = *se;
  unsigned q = 0;
#pragma unroll
  for (int r = 0; r < NV; ++r) {
    const unsigned h0 = fx_top(raw[r].x, emax), h1 = fx_top(raw[r].y, emax);
    q += h0 * h0 + h1 * h1;
  }
  if (q) atomicAdd(sq, (q >> 7) + 1u);
  __syncthreads();
  return FxScale{fx_scale(emax, *sq + 1u, M), emax == 0x7ff ? 0x7ff80000u : 0u};
}
WF_D fxc fx_from2(double2 d, FxScale f) { return fxc{fx_from(d.x, f.k), fx_from(d.y, f.k)}; }
// v 2^-(k + sh).  The power of two goes to the exponent field by an integer addition (values near the top
// of the range, where it could overflow, take a multiplication).
WF_D double fx_to(long long v, FxScale f, int sh = 0) {
  const int k = f.k + sh;
  double d = __ll2double_rn(v);
  if (k < -900) d *= fx_pow2(-k);
  else if (v != 0) d = __hiloint2double(__double2hiint(d) - (k << 20), __double2loint(d));
  return __hiloint2double(__double2hiint(d) | (int)f.nan, __double2loint(d));
}
WF_D double2 fx_to2(fxc v, FxScale f, int sh = 0) { return make_double2(fx_to(v.x, f, sh), fx_to(v.y, f, sh)); }
WF_D long long fx_rshift(long long v, int s) { return (v + (1ll << (s - 1))) >> s; }  // s >= 1, rounded

constexpr int fx_floor_log2(int n) { return n < 2 ? 0 : 1 + fx_floor_log2(n / 2); }
// the shift between a forward transform and the inverse that follows: ceil(log2(n) / 2), since the inverse's
// partial sums are below n ||z||_2, sqrt(n) times the forward's
constexpr int fx_mid(int n) { return (fx_floor_log2(n - 1) + 2) / 2; }

// slots of a tile of NL lines side by side; slots of one line with a pad per 8 (strided passes of
// neighbouring threads then fall on different banks)
template <int NL> struct ColMap {
  WF_D int operator()(int p) const { return p * NL; }
};
struct PadMap {
  WF_D int operator()(int p) const { return p + (p >> 3); }
};
constexpr int fx_padded(int m) { return m + m / 8; }

// twiddles exp(-2 pi i e / N), e < N, of the table exp(-2 pi i e / 2N) in shared memory
template <int N> WF_D void fx_load_tw(int4* tw, const int4* __restrict__ tab, int tid, int nt) {
  for (int e = tid; e < N; e += nt) tw[e] = __ldg(tab + 2 * e);
}

}  // namespace wf
