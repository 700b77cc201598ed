// wf_line.cuh -- transforms of one line held by a group of threads, exchanged through shared memory between
// two or three passes.  A line of M = R1 R2 R3 (R3 = 1: two passes) belongs to N1 = M / R1 threads; thread t
// enters with the elements n1 N1 + t in registers, so a caller loads them straight from memory, and the
// last pass hands its results out of registers.  Written over the complex type C (FP32 complex, or the
// 64-bit fixed point of wf_fix.cuh) with twiddles of type W.
#pragma once
#include "wf_common.cuh"

namespace wf {

// the engine's operations on FP32 complex values
template <int DIR> WF_D cx<float> ln_mul_i(cx<float> a) { return mul_si<DIR>(a); }
template <int DIR> WF_D cx<float> ln_twid(cx<float> a, float2 w) {
  return DIR < 0 ? cx<float>{a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x}
                 : cx<float>{a.x * w.x + a.y * w.y, a.y * w.x - a.x * w.y};
}
WF_D cx<float> ln_r2(cx<float> a) { return scale(a, 0.70710678118654752f); }
WF_D cx<float> ln_s3(cx<float> a) { return scale(a, 0.86602540378443865f); }
WF_D cx<float> ln_half(cx<float> a) { return scale(a, 0.5f); }
template <int DIR> WF_D cx<float> ln_rot9(cx<float> a, int m) {  // a exp(DIR 2 pi i m / 9), m = 1, 2, 4
  const float c = m == 1 ? 0.76604444311897804f : m == 2 ? 0.17364817766693035f : -0.93969262078590838f;
  const float s = m == 1 ? 0.64278760968653933f : m == 2 ? 0.98480775301220806f : 0.34202014332566873f;
  return ln_twid<DIR>(a, make_float2(c, -s));
}
template <int DIR, int m> WF_D cx<float> ln_rot16(cx<float> a) {  // a exp(DIR 2 pi i m / 16), m = 1, 3, 9
  const float c = m == 1 ? 0.92387953251128676f : m == 3 ? 0.38268343236508977f : -0.92387953251128676f;
  const float s = m == 1 ? 0.38268343236508977f : m == 3 ? 0.92387953251128676f : -0.38268343236508977f;
  return ln_twid<DIR>(a, make_float2(c, -s));
}
struct fxc;
template <int DIR> WF_D fxc ln_mul_i(fxc a);
template <int DIR> WF_D fxc ln_twid(fxc a, int4 w);
template <int DIR> WF_D fxc ln_rot9(fxc a, int m);

// ---- small DFTs in registers ---------------------------------------------------------------
template <class C> WF_D void ln_dft2(C& a, C& b) {
  const C s = a + b;
  b = a - b;
  a = s;
}
template <int DIR, class C> WF_D void ln_dft3(C& a, C& b, C& c) {
  const C t = b + c, u = b - c;
  const C m = a - ln_half(t), ju = ln_mul_i<DIR>(ln_s3(u));
  a = a + t;
  b = m + ju;
  c = m - ju;
}
template <int DIR, class C> WF_D void ln_dft4(C& a, C& b, C& c, C& d) {
  const C t0 = a + c, t1 = a - c, t2 = b + d, t3 = ln_mul_i<DIR>(b - d);
  a = t0 + t2;
  b = t1 + t3;
  c = t0 - t2;
  d = t1 - t3;
}
// v[0..RAD) -> its DFT in natural order
template <int RAD, int DIR, class C> WF_D void ln_dft(C* v) {
  if constexpr (RAD == 2) {
    ln_dft2(v[0], v[1]);
  } else if constexpr (RAD == 3) {
    ln_dft3<DIR>(v[0], v[1], v[2]);
  } else if constexpr (RAD == 4) {
    ln_dft4<DIR>(v[0], v[1], v[2], v[3]);
  } else if constexpr (RAD == 6) {
    // 2 x 3 without twiddles: n = 3 n1 + 2 n2, k = 3 k1 + 4 k2 (mod 6)
    C a0 = v[0], a1 = v[2], a2 = v[4], b0 = v[3], b1 = v[5], b2 = v[1];
    ln_dft3<DIR>(a0, a1, a2);
    ln_dft3<DIR>(b0, b1, b2);
    v[0] = a0 + b0;
    v[3] = a0 - b0;
    v[4] = a1 + b1;
    v[1] = a1 - b1;
    v[2] = a2 + b2;
    v[5] = a2 - b2;
  } else if constexpr (RAD == 8) {
    ln_dft4<DIR>(v[0], v[2], v[4], v[6]);
    ln_dft4<DIR>(v[1], v[3], v[5], v[7]);
    // W8^1 = (1 + DIR i)/sqrt2, W8^2 = DIR i, W8^3 = (-1 + DIR i)/sqrt2
    const C o1 = ln_r2(v[3] + ln_mul_i<DIR>(v[3])), o2 = ln_mul_i<DIR>(v[5]), o3 = ln_r2(ln_mul_i<DIR>(v[7]) - v[7]);
    const C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
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
    ln_dft3<DIR>(v[0], v[3], v[6]);
    ln_dft3<DIR>(v[1], v[4], v[7]);
    ln_dft3<DIR>(v[2], v[5], v[8]);
    v[4] = ln_rot9<DIR>(v[4], 1);
    v[5] = ln_rot9<DIR>(v[5], 2);
    v[7] = ln_rot9<DIR>(v[7], 2);
    v[8] = ln_rot9<DIR>(v[8], 4);
    ln_dft3<DIR>(v[0], v[1], v[2]);
    ln_dft3<DIR>(v[3], v[4], v[5]);
    ln_dft3<DIR>(v[6], v[7], v[8]);
    C t = v[1];  // transpose the 3 x 3 result
    v[1] = v[3];
    v[3] = t;
    t = v[2];
    v[2] = v[6];
    v[6] = t;
    t = v[5];
    v[5] = v[7];
    v[7] = t;
  } else if constexpr (RAD == 16) {
    // 4 x 4: columns n = 4 n1 + n2, twiddles W16^(n2 k1), rows; k = k1 + 4 k2
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) ln_dft4<DIR>(v[n2], v[4 + n2], v[8 + n2], v[12 + n2]);
    v[5] = ln_rot16<DIR, 1>(v[5]);
    v[6] = ln_r2(v[6] + ln_mul_i<DIR>(v[6]));
    v[7] = ln_rot16<DIR, 3>(v[7]);
    v[9] = ln_r2(v[9] + ln_mul_i<DIR>(v[9]));
    v[10] = ln_mul_i<DIR>(v[10]);
    v[11] = ln_r2(ln_mul_i<DIR>(v[11]) - v[11]);
    v[13] = ln_rot16<DIR, 3>(v[13]);
    v[14] = ln_r2(ln_mul_i<DIR>(v[14]) - v[14]);
    v[15] = ln_rot16<DIR, 9>(v[15]);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) ln_dft4<DIR>(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = i + 1; j < 4; ++j) {
        const C t = v[4 * i + j];
        v[4 * i + j] = v[4 * j + i];
        v[4 * j + i] = t;
      }
  } else {
    static_assert(RAD == 12, "radix");
    // 4 x 3 without twiddles: n = 3 n1 + 4 n2, k = 9 k1 + 4 k2 (mod 12)
    C a[3][4];
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < 4; ++n1) a[n2][n1] = v[(3 * n1 + 4 * n2) % 12];
      ln_dft4<DIR>(a[n2][0], a[n2][1], a[n2][2], a[n2][3]);
    }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      ln_dft3<DIR>(a[0][k1], a[1][k1], a[2][k1]);
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) v[(9 * k1 + 4 * k2) % 12] = a[k2][k1];
    }
  }
}

struct LnNone {
  WF_D void operator()(int) const {}
};

// Forward transform, a multiplier at each k, and the inverse transform (unnormalised) of one line held
// by TPL = M / R1 threads: thread t enters with v[n1] = z[n1 (M / R1) + t] and leaves with the same
// elements of the result.  n = n1 R2 R3 + n2 R3 + n3, k = k1 + R1 k2 + R1 R2 k3; every pass writes the
// slots it read, so one barrier stands between two passes.  s: the line's M slots (slot p at
// s[map(p)]); tw[e] = digits of exp(-2 pi i e / M); ph(k, X): the multiplier.  Every thread of the CTA
// calls it; all of the CTA's lines are done together.
template <int M, class PL, class C, class W, class MAP, class PH>
WF_D void ln_convolve(C (&v)[PL::r1], C* s, const MAP& map, int t, const W* tw, const PH& ph) {
  constexpr int R1 = PL::r1, R2 = PL::r2, R3 = PL::r3, N1 = M / R1;
  static_assert(R1 * R2 * R3 == M, "plan");
  ln_dft<R1, -1>(v);
  s[map(t)] = v[0];
#pragma unroll
  for (int k1 = 1; k1 < R1; ++k1) s[map(k1 * N1 + t)] = ln_twid<-1>(v[k1], tw[t * k1]);
  __syncthreads();
  if constexpr (R3 > 1) {
    for (int j = t; j < M / R2; j += N1) {
      const int k1 = j / R3, n3 = j % R3, base = k1 * R2 * R3 + n3;
      C a[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) a[n2] = s[map(base + n2 * R3)];
      ln_dft<R2, -1>(a);
      s[map(base)] = a[0];
#pragma unroll
      for (int k2 = 1; k2 < R2; ++k2) s[map(base + k2 * R3)] = ln_twid<-1>(a[k2], tw[R1 * n3 * k2]);
    }
    __syncthreads();
    for (int j = t; j < M / R3; j += N1) {
      const int k1 = j / R2, k2 = j % R2, base = j * R3;
      C a[R3];
#pragma unroll
      for (int n3 = 0; n3 < R3; ++n3) a[n3] = s[map(base + n3)];
      ln_dft<R3, -1>(a);
#pragma unroll
      for (int k3 = 0; k3 < R3; ++k3) a[k3] = ph(k1 + R1 * k2 + R1 * R2 * k3, a[k3]);
      ln_dft<R3, +1>(a);
      s[map(base)] = a[0];
#pragma unroll
      for (int n3 = 1; n3 < R3; ++n3) s[map(base + n3)] = ln_twid<+1>(a[n3], tw[R1 * n3 * k2]);
    }
    __syncthreads();
    for (int j = t; j < M / R2; j += N1) {
      const int k1 = j / R3, n3 = j % R3, base = k1 * R2 * R3 + n3;
      C a[R2];
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) a[k2] = s[map(base + k2 * R3)];
      ln_dft<R2, +1>(a);
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) s[map(base + n2 * R3)] = ln_twid<+1>(a[n2], tw[(n2 * R3 + n3) * k1]);
    }
  } else {
    for (int j = t; j < R1; j += N1) {  // j = k1
      C a[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) a[n2] = s[map(j * R2 + n2)];
      ln_dft<R2, -1>(a);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) a[k2] = ph(j + R1 * k2, a[k2]);
      ln_dft<R2, +1>(a);
      s[map(j * R2)] = a[0];
#pragma unroll
      for (int n2 = 1; n2 < R2; ++n2) s[map(j * R2 + n2)] = ln_twid<+1>(a[n2], tw[n2 * j]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) v[k1] = s[map(k1 * N1 + t)];
  ln_dft<R1, +1>(v);
}

// The forward half alone, in either direction (DIR = +1: conjugate twiddles): enters like ln_convolve
// and hands every Z_k the thread ends with to out(k, Z_k, i), i = 0, 1, ... its number in
// the thread (k = ln_index(t, i)).  pre(m) runs before the m-th round of the
// last pass, whose results are m RL ... m RL + RL - 1, RL = PL's last radix (a place to start loads that out uses).  TWS: W_M^e = tw[TWS e].
template <int M, class PL, int DIR, int TWS = 1, class C, class W, class MAP, class OUT, class PRE = LnNone>
WF_D void ln_forward(C (&v)[PL::r1], C* s, const MAP& map, int t, const W* tw, const OUT& out, const PRE& pre = PRE()) {
  constexpr int R1 = PL::r1, R2 = PL::r2, R3 = PL::r3, N1 = M / R1;
  ln_dft<R1, DIR>(v);
  s[map(t)] = v[0];
#pragma unroll
  for (int k1 = 1; k1 < R1; ++k1) s[map(k1 * N1 + t)] = ln_twid<DIR>(v[k1], tw[TWS * t * k1]);
  __syncthreads();
  if constexpr (R3 > 1) {
    for (int j = t; j < M / R2; j += N1) {
      const int k1 = j / R3, n3 = j % R3, base = k1 * R2 * R3 + n3;
      C a[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) a[n2] = s[map(base + n2 * R3)];
      ln_dft<R2, DIR>(a);
      s[map(base)] = a[0];
#pragma unroll
      for (int k2 = 1; k2 < R2; ++k2) s[map(base + k2 * R3)] = ln_twid<DIR>(a[k2], tw[TWS * R1 * n3 * k2]);
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < (M / R3 + N1 - 1) / N1; ++m) {
      const int j = t + m * N1;
      if ((M / R3) % N1 == 0 || j < M / R3) {
        pre(m);
        C a[R3];
#pragma unroll
        for (int n3 = 0; n3 < R3; ++n3) a[n3] = s[map(j * R3 + n3)];
        ln_dft<R3, DIR>(a);
#pragma unroll
        for (int k3 = 0; k3 < R3; ++k3) out(j / R2 + R1 * (j % R2) + R1 * R2 * k3, a[k3], m * R3 + k3);
      }
    }
  } else {
#pragma unroll
    for (int m = 0; m < (R1 + N1 - 1) / N1; ++m) {
      const int j = t + m * N1;
      if (R1 % N1 == 0 || j < R1) {
        pre(m);
        C a[R2];
#pragma unroll
        for (int n2 = 0; n2 < R2; ++n2) a[n2] = s[map(j * R2 + n2)];
        ln_dft<R2, DIR>(a);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) out(j + R1 * k2, a[k2], m * R2 + k2);
      }
    }
  }
}

// The same with the result left in the line's slots in natural order (a barrier after it).
template <int M, class PL, int DIR, int TWS, class C, class W, class MAP>
WF_D void ln_forward_nat(C (&v)[PL::r1], C* s, const MAP& map, int t, const W* tw) {
  constexpr int R1 = PL::r1, R2 = PL::r2, R3 = PL::r3, N1 = M / R1;
  constexpr int RL = R3 > 1 ? R3 : R2, NB = M / RL, PER = (NB + N1 - 1) / N1;
  C res[PER * RL];
  ln_forward<M, PL, DIR, TWS>(v, s, map, t, tw, [&](int, C X, int i) { res[i] = X; });
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
template <int M, class PL, int DIR, int TWS = 1, class C, class W, class MAP, class IN>
WF_D void ln_inverse(C (&v)[PL::r1], C* s, const MAP& map, int t, const W* tw, const IN& in) {
  constexpr int R1 = PL::r1, R2 = PL::r2, R3 = PL::r3, N1 = M / R1;
  constexpr int RL = R3 > 1 ? R3 : R2, NB = M / RL, PER = (NB + N1 - 1) / N1;
  C a[PER][RL];
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
      ln_dft<RL, DIR>(a[m]);
      const int e = R3 > 1 ? R1 * (j % R2) : j;  // twiddle step of output r
      s[map(j * RL)] = a[m][0];
#pragma unroll
      for (int r = 1; r < RL; ++r) s[map(j * RL + r)] = ln_twid<DIR>(a[m][r], tw[TWS * r * e]);
    }
  }
  __syncthreads();
  if constexpr (R3 > 1) {
    for (int j = t; j < M / R2; j += N1) {
      const int k1 = j / R3, n3 = j % R3, base = k1 * R2 * R3 + n3;
      C b[R2];
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) b[k2] = s[map(base + k2 * R3)];
      ln_dft<R2, DIR>(b);
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) s[map(base + n2 * R3)] = ln_twid<DIR>(b[n2], tw[TWS * (n2 * R3 + n3) * k1]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) v[k1] = s[map(k1 * N1 + t)];
  ln_dft<R1, DIR>(v);
}

// the k of the i-th result of thread t in ln_forward
template <int M, class PL> WF_D int ln_index(int t, int i) {
  constexpr int RL = PL::r3 > 1 ? PL::r3 : PL::r2;
  const int j = t + (i / RL) * (M / PL::r1), r = i % RL;
  return PL::r3 > 1 ? j / PL::r2 + PL::r1 * (j % PL::r2) + PL::r1 * PL::r2 * r : j + PL::r1 * r;
}

// Slots of a tile of NL lines side by side, and slots of one line on its own with a pad slot per 8 (or per 16
// where the last pass strides by 16): strided accesses of neighbouring threads then fall on different banks.
template <int NL> struct ColMap {
  WF_D int operator()(int p) const { return p * NL; }
};
template <int SH = 3> struct PadMapT {
  WF_D int operator()(int p) const { return p + (p >> SH); }
};
using PadMap = PadMapT<3>;
// slots of a padded line of m elements held by n1 threads: its length modulo `banks` elements (the elements of one
// shared-memory wavefront) is n1, so that the next line's threads continue on the banks behind this one's
constexpr int ln_padded(int m, int sh, int n1, int banks) {
  int l = m + (m >> sh);
  while (n1 < banks && l % banks != n1 % banks) ++l;
  return l;
}

// Sum over the CTA of the threads' double-float accumulators; valid in thread 0.  Each warp adds its 32 values
// exactly, as integers in units of 2^-57 of the largest (three reductions of limbs), and only the warps' sums
// meet in FP64: a tree of FP64 shuffles over all threads keeps GB300's FP64 pipe busy for ~1 us per CTA.
// The result does not depend on any order.  red holds >= 32 doubles.
WF_D long long acc_fixed(float f, int E) {  // f 2^(33 - (E - 150)) truncated, for exponents up to E
  const unsigned u = __float_as_uint(f);
  const int e = (u >> 23) & 0xff, sh = 33 - (E - e);
  const long long m = e ? (long long)((u & 0x7fffffu) | 0x800000u) : 0;
  const long long v = sh >= 0 ? m << sh : (sh > -24 ? m >> -sh : 0);
  return (int)u < 0 ? -v : v;
}
WF_D double block_sum_acc(const AccF& a, double* red) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5, nl = warp_lanes();
  const unsigned mask = lane_mask(nl);
  const int E = (int)(__reduce_max_sync(mask, __float_as_uint(a.hi) & 0x7fffffffu) >> 23);
  const long long v = acc_fixed(a.hi, E) + acc_fixed(a.lo, E);
  const int s0 = __reduce_add_sync(mask, (int)(v & 0x1fffff));
  const int s1 = __reduce_add_sync(mask, (int)((v >> 21) & 0x1fffff));
  const int s2 = __reduce_add_sync(mask, (int)(v >> 42));
  long long* sums = reinterpret_cast<long long*>(red);
  __shared__ int exps[32];
  __syncthreads();
  if (l == 0) {
    sums[w] = (long long)s0 + ((long long)s1 << 21) + ((long long)s2 << 42);
    exps[w] = E;
  }
  __syncthreads();
  double r = 0.0;
  if (w == 0) {
    for (int i = l; i < nw; i += nl) {  // one round but in a CTA of a single partial warp
      const int k = exps[i] - 150 - 33;  // the units; a non-finite accumulator makes the sum a NaN
      r += exps[i] == 0xff ? __longlong_as_double(0x7ff8000000000000ll)
                           : __ll2double_rn(sums[i]) * __hiloint2double((k + 1023) << 20, 0);
    }
    for (int o = 16; o > 0; o >>= 1)
      if (o < nw) {
        const double t = __shfl_down_sync(mask, r, o);
        if (l + o < nl) r += t;
      }
  }
  return r;
}

}  // namespace wf
