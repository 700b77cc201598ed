// wf_line.cuh -- transforms of one line held by a group of threads, exchanged through shared memory between
// two or three passes.  A line of M = R1 R2 R3 (R3 = 1: two passes) belongs to N1 = M / R1 threads; thread t
// enters with the elements n1 N1 + t in registers, so a caller loads them straight from memory, and the
// last pass hands its results out of registers.  Written over the complex type C (the 64-bit fixed point of
// wf_fix.cuh) with twiddles of type W.
#pragma once
#include "wf_common.cuh"

namespace wf {

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

}  // namespace wf
