// wf_lines32.cuh -- the FP32 CG passes on the line engine (wf_line.cuh).  A CTA's threads load their elements of r,
// p, x or T straight into registers (rows of NL consecutive kz columns), exchange once or twice through
// shared memory inside the transform and store from registers: two to four shared-memory accesses per
// element where a tile staged through shared memory took six or more, and no barrier around the loads.
//
// c(k) comes from an octant table [N/2+1][N/2+1][N/2] over (|ky|, |kx|, kz), built once per inner solve: a row of
// NL columns is one or two sectors.  Gathering c by n^2 touches a sector per element; at 512^3 those gathers
// moved as many bytes from L2 as the spectra themselves.
//
// Memory bounds these passes; per launch at 512^3, before (staged tiles) and now, of the time their bytes take at the
// measured copy rate of 6.67 TB/s:
//   x pass 1 (six spectra)            0.70 -> 0.61 ms   79%
//   x pass 2 (four)                   0.58 -> 0.45      72%
//   coarse x stage (two)              0.41 -> 0.23      70%
//   z turn (two and D)                0.43 -> 0.39      61%
//   coarse z stage (one and D)        0.38 -> 0.31      52%
//   y pass (two)                      0.21 -> 0.17      94%   (its tensor-copied tiles, of rows of 128 bytes)
// A solve at 512^3: 349 -> 292 ms, at 144^3: 10.4 -> 8.8 ms.
#pragma once
#include "wf_line.cuh"
#include "wf_spectral.cuh"

namespace wf {

template <int A, int B, int C> struct LnRad {
  static constexpr int r1 = A, r2 = B, r3 = C;
};
template <int M> struct F32Plan { using T = LnRad<0, 0, 0>; };
#define WF_PLAN(M, A, B, C) \
  template <> struct F32Plan<M> { using T = LnRad<A, B, C>; }
WF_PLAN(8, 4, 2, 1);
WF_PLAN(12, 3, 4, 1);
WF_PLAN(16, 4, 4, 1);
WF_PLAN(24, 4, 6, 1);
WF_PLAN(32, 8, 4, 1);
WF_PLAN(36, 6, 6, 1);
WF_PLAN(48, 6, 8, 1);
WF_PLAN(54, 6, 9, 1);
WF_PLAN(64, 8, 8, 1);
WF_PLAN(72, 8, 9, 1);
WF_PLAN(96, 8, 12, 1);
WF_PLAN(108, 9, 12, 1);
WF_PLAN(128, 16, 8, 1);
WF_PLAN(144, 12, 12, 1);
WF_PLAN(192, 12, 16, 1);
WF_PLAN(216, 6, 6, 6);
WF_PLAN(256, 16, 16, 1);
WF_PLAN(288, 6, 6, 8);
WF_PLAN(384, 6, 8, 8);
WF_PLAN(512, 8, 8, 8);
#undef WF_PLAN

// plan of the x passes: small butterflies (their vector updates need the registers)
template <int M> struct F32XPlan { using T = typename F32Plan<M>::T; };
#define WF_PLAN(M, A, B, C) \
  template <> struct F32XPlan<M> { using T = LnRad<A, B, C>; }
WF_PLAN(96, 8, 4, 3);
WF_PLAN(108, 9, 4, 3);
WF_PLAN(128, 8, 4, 4);
WF_PLAN(144, 6, 6, 4);
WF_PLAN(192, 8, 6, 4);
WF_PLAN(256, 8, 8, 4);
WF_PLAN(288, 12, 6, 4);
WF_PLAN(384, 12, 8, 4);
WF_PLAN(512, 16, 8, 4);
#undef WF_PLAN

// the largest divisor of n up to cap, of those that are multiples of 4 (rows of whole 32-byte sectors) if any
constexpr int div_sector(int n, int cap) {
  for (int d = cap - cap % 4; d >= 4; d -= 4)
    if (n % d == 0) return d;
  return div_le(n, cap);
}
// Geometry of an x or y pass: NL columns (a divisor of N/2, at most NLMAX) by N rows, with at most TMAX threads
template <int N_, int NLMAX, int TMAX, int MINB_ = 0, class PL_ = typename F32Plan<N_>::T, int EARLY_ = 0> struct LX {
  using PL = PL_;
  using C = cx<float>;
  static constexpr int N = N_, NH = N / 2, R1 = PL::r1, N1 = N / R1;
  static constexpr int NL = div_sector(NH, cmin(NLMAX, TMAX / N1));
  static constexpr int NT = NL * N1, KB = NH / NL;
  static constexpr int YP = (N / 2 / (NL / 2) + KB) / KB;  // rows of CTAs for the pairs ky = 0 .. N/2 of column 0
  static constexpr int MINB = MINB_ < 0 ? cmin(16, -MINB_ / NT) : MINB_;  // < 0: so many threads per SM
  static constexpr int RL = PL::r3 > 1 ? PL::r3 : PL::r2;
  static constexpr int EARLY = EARLY_;  // x pass 2: results per thread up to which r and p are requested at the start
  static constexpr size_t SMEM = (size_t)(N * NL + N) * sizeof(C);
  static constexpr size_t OCT = (size_t)(NH + 1) * (NH + 1) * NH;    // entries of the octant table
  static_assert(PL::r1 * PL::r2 * PL::r3 == N && NL >= 2, "plan");
};
template <int N> WF_D const float* oct_row(const float* oct, int ky_s, int kxs) {
  constexpr int NH = N / 2;
  return oct + ((size_t)(ky_s < 0 ? -ky_s : ky_s) * (NH + 1) + (kxs < 0 ? -kxs : kxs)) * NH;
}
// oct[z][|ky|][|kx|][kz] = c(n^2).  grid (N/2 + 1, N/2 + 1, systems)
template <int N>
__global__ void k_oct(const float* __restrict__ ctab, float* __restrict__ oct, size_t octs, int tabs,
                      const CgScal* __restrict__ sc) {
  constexpr int NH = N / 2;
  const int z = blockIdx.z, ky = blockIdx.y, kx = blockIdx.x;
  if (sc[z].done) return;
  float* o = oct + z * octs + ((size_t)ky * (NH + 1) + kx) * NH;
  for (int kz = threadIdx.x; kz < NH; kz += blockDim.x) o[kz] = ctab[(size_t)z * tabs + kx * kx + ky * ky + kz * kz];
}
template <int N> WF_D void ln_load_tw(float2* tw, const float2* __restrict__ tab, int tid, int nt) {
  for (int e = tid; e < N; e += nt) tw[e] = __ldg(tab + 2 * e);
}
WF_D cx<float> ld2(const float2* p) {
  const float2 v = *p;
  return cx<float>{v.x, v.y};
}
WF_D void st2(float2* p, cx<float> v) { *p = make_float2(v.x, v.y); }

// x pass 1:  p_new = r + beta p_old;  x += alpha_prev p_old;  T = IFFT_x(c (.) p_new);  partial of <p_new, m p_new>
// (the work and the sums of k_cg_xinv; the packed column takes its partner element at -k in registers).
// Rows of 16 columns (128 bytes): rows of 64 bytes a megabyte apart copy at 3.2 TB/s, these at 6.6.  Two CTAs of 512
// threads per SM (64 registers; 0.81 ms with one).  grid (N/2 / NL, N, systems)
template <class G, bool UNIT_M>
__global__ void __launch_bounds__(G::NT, G::MINB)
k_ln_xinv(const float2* __restrict__ r, float2* P0, float2* P1, float2* __restrict__ x, float2* __restrict__ T,
          const float* __restrict__ oct, const float* __restrict__ ctab, const float* __restrict__ mtab,
          const float2* __restrict__ twtab, double* __restrict__ partials, const CgScal* __restrict__ sc, Bat bt) {
  using C = cx<float>;
  constexpr int N = G::N, NH = G::NH, NL = G::NL, R1 = G::R1, N1 = G::N1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  C* slots = reinterpret_cast<C*>(smem_raw);
  float2* tw = reinterpret_cast<float2*>(slots + N * NL);
  __shared__ double red[32];
  const int z = blockIdx.z, tid = threadIdx.x, l = tid % NL, t = tid / NL;
  ln_load_tw<N>(tw, twtab, tid, G::NT);
  chain_start();
  sc += z;
  if (finished(sc)) return;
  const float2* __restrict__ pold = ((sc->lit & 1) ? P1 : P0) + z * bt.spec;
  float2* __restrict__ pnew = ((sc->lit & 1) ? P0 : P1) + z * bt.spec;
  r += z * bt.spec;
  x += z * bt.spec;
  T += z * bt.spec;
  oct += z * G::OCT;
  ctab += z * bt.tab;
  mtab += z * bt.tab;
  const float beta = (float)sc->beta, alpha = (float)sc->alpha_prev;
  const int ky = blockIdx.y, ky_s = sfreq(ky, N), kz = blockIdx.x * NL + l;
  const size_t rowstride = (size_t)N * NH, base = (size_t)ky * NH + kz;
  AccF acc;  // the terms are >= 0: a chunk's terms are summed in FP32 first
  C v[R1];
  constexpr int CH = R1 % 4 == 0 ? (R1 > 8 ? 2 : 4) : 3;  // elements whose loads are in flight together
  static_assert(R1 % CH == 0, "chunks");
#pragma unroll
  for (int q0 = 0; q0 < R1; q0 += CH) {
    C rv[CH], po[CH], xv[CH];
    float cv[CH], part = 0.f;
#pragma unroll
    for (int j = 0; j < CH; ++j) {
      const int kx = (q0 + j) * N1 + t;
      const size_t e = base + (size_t)kx * rowstride;
      rv[j] = ld2(r + e);
      po[j] = ld2(pold + e);
      xv[j] = ld2(x + e);
      cv[j] = oct_row<N>(oct, ky_s, sfreq(kx, N))[kz];
    }
#pragma unroll
    for (int j = 0; j < CH; ++j) {
      const int kx = (q0 + j) * N1 + t;
      const size_t e = base + (size_t)kx * rowstride;
      const C p{rv[j].x + beta * po[j].x, rv[j].y + beta * po[j].y};
      st2(pnew + e, p);
      st2(x + e, C{xv[j].x + alpha * po[j].x, xv[j].y + alpha * po[j].y});
      const float s2 = 2.f * (p.x * p.x + p.y * p.y);
      if (UNIT_M) {
        part += s2;
      } else {
        const int kxs = sfreq(kx, N);
        part += mtab[kxs * kxs + ky_s * ky_s + kz * kz] * s2;
      }
      const float c = kz == 0 ? 1.f : cv[j];  // column 0 stays raw for the pair below
      v[q0 + j] = C{c * p.x, c * p.y};
    }
    if (kz != 0) acc.add(part);
  }
  if (kz == 0) {  // packed column: c and m act on the planes P0 = (Z + conj Z(-k)) / 2, PN = (Z - conj Z(-k)) / 2i
#pragma unroll
    for (int q0 = 0; q0 < R1; q0 += CH) {
      C rq[CH], pq[CH];
#pragma unroll
      for (int j = 0; j < CH; ++j) {
        const int kx = (q0 + j) * N1 + t;
        const size_t eq = (size_t)((N - ky) % N) * NH + (size_t)((N - kx) % N) * rowstride;
        rq[j] = ld2(r + eq);
        pq[j] = ld2(pold + eq);
      }
      float part = 0.f;
#pragma unroll
      for (int j = 0; j < CH; ++j) {
        const int kxs = sfreq((q0 + j) * N1 + t, N), n2 = kxs * kxs + ky_s * ky_s;
        const C p = v[q0 + j];
        const float qx = rq[j].x + beta * pq[j].x, qy = rq[j].y + beta * pq[j].y;
        const float a0 = 0.5f * (p.x + qx), b0 = 0.5f * (p.y - qy), aN = 0.5f * (p.y + qy), bN = 0.5f * (qx - p.x);
        part += mtab[n2] * (a0 * a0 + b0 * b0) + mtab[n2 + NH * NH] * (aN * aN + bN * bN);
        const float c = ctab[n2], cN = ctab[n2 + NH * NH], a = 0.5f * (c + cN), b = 0.5f * (c - cN);
        v[q0 + j] = C{a * p.x + b * qx, a * p.y - b * qy};
      }
      acc.add(part);
    }
  }
  __syncthreads();  // twiddles
  ln_forward<N, typename G::PL, +1>(v, slots + l, ColMap<NL>{}, t, tw,
                                    [&](int k, C X, int) { st2(T + base + (size_t)k * rowstride, X); });
  const double sum = block_sum_acc(acc, red);
  if (tid == 0) partials[(size_t)z * bt.part + blockIdx.y * gridDim.x + blockIdx.x] = sum;
}

// x stage of the coarse projection:  T = IFFT_x(c (.) r).  With n3 > 0 the first row of CTAs takes beta and the stop
// test of the iteration before from its n3 pairs of partial sums.  grid (N/2 / NL, N + (n3 > 0), systems)
template <class G>
__global__ void __launch_bounds__(G::NT, G::MINB)
k_ln_xcr(const float2* __restrict__ r, float2* __restrict__ T, const float* __restrict__ oct,
         const float* __restrict__ ctab, const float2* __restrict__ twtab, CgScal* __restrict__ sc, Bat bt,
         const double* __restrict__ part, int n3, double inv_vc) {
  using C = cx<float>;
  constexpr int N = G::N, NH = G::NH, NL = G::NL, R1 = G::R1, N1 = G::N1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  C* slots = reinterpret_cast<C*>(smem_raw);
  float2* tw = reinterpret_cast<float2*>(slots + N * NL);
  const int z = blockIdx.z, tid = threadIdx.x, l = tid % NL, t = tid / NL;
  ln_load_tw<N>(tw, twtab, tid, G::NT);
  chain_start();
  if (finished(sc + z)) return;
  int ky = blockIdx.y;
  if (n3 > 0 && ky-- == 0) {
    if (blockIdx.x == 0)
      fin_beta(part + (size_t)z * bt.part, n3, inv_vc, sc + z, reinterpret_cast<double*>(smem_raw));
    return;
  }
  r += z * bt.spec;
  T += z * bt.spec;
  oct += z * G::OCT;
  ctab += z * bt.tab;
  const int ky_s = sfreq(ky, N), kz = blockIdx.x * NL + l;
  const size_t rowstride = (size_t)N * NH, base = (size_t)ky * NH + kz;
  C v[R1];
  float cv[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q) {
    const int kx = q * N1 + t;
    v[q] = ld2(r + base + (size_t)kx * rowstride);
    cv[q] = oct_row<N>(oct, ky_s, sfreq(kx, N))[kz];
  }
  if (kz != 0) {
#pragma unroll
    for (int q = 0; q < R1; ++q) v[q] = scale(v[q], cv[q]);
  } else {  // packed column: the pair of multipliers with the element at -k
#pragma unroll
    for (int q = 0; q < R1; ++q) {
      const int kx = q * N1 + t, kxs = sfreq(kx, N);
      const C rq = ld2(r + (size_t)((N - ky) % N) * NH + (size_t)((N - kx) % N) * rowstride);
      const float cN = ctab[kxs * kxs + ky_s * ky_s + NH * NH], a = 0.5f * (cv[q] + cN), b = 0.5f * (cv[q] - cN);
      v[q] = C{a * v[q].x + b * rq.x, a * v[q].y - b * rq.y};
    }
  }
  __syncthreads();
  ln_forward<N, typename G::PL, +1>(v, slots + l, ColMap<NL>{}, t, tw,
                                    [&](int k, C X, int) { st2(T + base + (size_t)k * rowstride, X); });
}

// x pass 2:  T^ = FFT_x(T);  q = m p + c T^;  r -= alpha q;  partials of <r, r> and of the residual estimate (the
// work and the sums of k_cg_xupd, two per CTA).  The packed column pairs a line with the one at -ky: the CTAs
// behind the first N rows of CTAs take column 0 of NL / 2 such pairs each (ky <= N/2), the others skip it.  p, r
// and c of up to eight results are requested before their butterflies.  grid (KB, N + YP, systems)
template <class G, bool UNIT_M>
__global__ void __launch_bounds__(G::NT, G::MINB)
k_ln_xupd(const float2* __restrict__ T, float2* __restrict__ r, const float2* P0, const float2* P1,
          const float* __restrict__ oct, const float* __restrict__ ctab, const float* __restrict__ mtab,
          const float2* __restrict__ twtab, double* __restrict__ partials, const CgScal* __restrict__ sc, Bat bt) {
  using C = cx<float>;
  using PL = typename G::PL;
  constexpr int N = G::N, NH = G::NH, NL = G::NL, R1 = G::R1, N1 = G::N1, RL = G::RL;
  // rounds whose operands are requested together: all of them with the T loads where they are few (EARLY: one
  // trip to memory instead of two, which is what a small grid's pass waits for), else up to eight results
  constexpr int ROUNDS = (N / RL + N1 - 1) / N1;
  constexpr bool EARLY = ROUNDS * RL <= G::EARLY;
  constexpr int PD = EARLY ? ROUNDS : cmin(ROUNDS, RL <= 4 ? 2 : 1);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  C* slots = reinterpret_cast<C*>(smem_raw);
  float2* tw = reinterpret_cast<float2*>(slots + N * NL);
  __shared__ double red[32];
  const int z = blockIdx.z, tid = threadIdx.x, l = tid % NL, t = tid / NL;
  ln_load_tw<N>(tw, twtab, tid, G::NT);
  chain_start();
  sc += z;
  if (finished(sc)) return;
  const bool pair = blockIdx.y >= N;
  const int first = ((blockIdx.y - N) * G::KB + blockIdx.x) * (NL / 2);  // a pair CTA's first ky
  partials += (size_t)z * bt.part + 2 * (blockIdx.y * G::KB + blockIdx.x);
  if (pair && first > N / 2) {
    if (tid < 2) partials[tid] = 0.0;
    return;
  }
  // a pair CTA's line slots 2 j and 2 j + 1 hold column 0 at ky and -ky
  const int ky = pair ? first + l / 2 : blockIdx.y;
  const bool live = !pair || (ky <= N / 2 && l < NL / 2 * 2);
  const float2* __restrict__ p = ((sc->lit & 1) ? P0 : P1) + z * bt.spec;  // this iteration's p_new
  T += z * bt.spec;
  r += z * bt.spec;
  oct += z * G::OCT;
  ctab += z * bt.tab;
  mtab += z * bt.tab;
  const float alpha = (float)sc->alpha;
  const int ky_s = sfreq(ky, N);
  const size_t rowstride = (size_t)N * NH;
  const int row_y = pair && l % 2 == 1 ? (N - ky) % N : ky;
  const size_t base = (size_t)row_y * NH + (pair ? 0 : blockIdx.x * NL + l);
  C v[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q) v[q] = live ? ld2(T + base + (size_t)(q * N1 + t) * rowstride) : C{0.f, 0.f};
  const int kz = pair ? 0 : blockIdx.x * NL + l;
  C rv[PD * RL], pv[PD * RL];
  float cv[PD * RL];
  auto request = [&](int m) {
#pragma unroll
    for (int j = 0; j < PD * RL; ++j) {
      if ((N / RL) % N1 != 0 && t + (m + j / RL) * N1 >= N / RL) continue;
      const int k = ln_index<N, PL>(t, m * RL + j);
      const size_t e = base + (size_t)k * rowstride;
      rv[j] = ld2(r + e);
      pv[j] = ld2(p + e);
      cv[j] = oct_row<N>(oct, ky_s, sfreq(k, N))[kz];
    }
  };
  if (EARLY && !pair) request(0);
  __syncthreads();
  AccF a_rr, a_rc;
  if (!pair) {
    float s_rr = 0.f, s_rc = 0.f;
    ln_forward<N, PL, -1>(
        v, slots + l, ColMap<NL>{}, t, tw,
        [&](int k, C X, int i) {
          if (kz == 0) return;
          const int j = i % (PD * RL);
          float m = 1.f;
          if (!UNIT_M) {
            const int kxs = sfreq(k, N);
            m = mtab[kxs * kxs + ky_s * ky_s + kz * kz];
          }
          const float c = cv[j];
          rv[j].x -= alpha * (m * pv[j].x + c * X.x);
          rv[j].y -= alpha * (m * pv[j].y + c * X.y);
          st2(r + base + (size_t)k * rowstride, rv[j]);
          const float m2 = 2.f * (rv[j].x * rv[j].x + rv[j].y * rv[j].y);
          s_rr += m2;
          s_rc += m2 * __frcp_rn(c * c);
          if (i % 2 == 1 || i % RL == RL - 1) {  // the terms are >= 0: two elements' are summed in FP32 first
            a_rr.add(s_rr);
            a_rc.add(s_rc);
            s_rr = s_rc = 0.f;
          }
        },
        [&](int m) {
          if (!EARLY && m % PD == 0) request(m);
        });
  } else {
    // p, r and the tables are asked for before the transform where they fit the registers (a small grid's pass waits
    // for these CTAs; the launch at 64^3 13.5 -> 11.7 us, the solve 4.08 -> 3.95 ms)
    constexpr bool AHEAD = R1 <= 8;
    constexpr int NK = AHEAD ? R1 : 1;
    const bool mine = live && !(l % 2 == 1 && row_y == ky);
    C pk[NK], rk[NK];
    float c0k[NK], cNk[NK];
    auto ask = [&](int j, int k) {
      const int kxs = sfreq(k, N), n2 = kxs * kxs + ky_s * ky_s;
      pk[j] = ld2(p + base + (size_t)k * rowstride);
      rk[j] = ld2(r + base + (size_t)k * rowstride);
      c0k[j] = ctab[n2];
      cNk[j] = ctab[n2 + NH * NH];
    };
    if (AHEAD && mine) {
#pragma unroll
      for (int j = 0; j < NK; ++j) ask(j, t + j * N1);
    }
    ln_forward_nat<N, PL, -1, 1>(v, slots + l, ColMap<NL>{}, t, tw);  // T^ of both lines in natural order
    auto update = [&](int j, int k) {
      const int kxs = sfreq(k, N), n2 = kxs * kxs + ky_s * ky_s;
      const float c0 = c0k[j], cN = cNk[j], m0 = mtab[n2], mN = mtab[n2 + NH * NH];
      const float ca = 0.5f * (c0 + cN), cb = 0.5f * (c0 - cN), ma = 0.5f * (m0 + mN), mb = 0.5f * (m0 - mN);
      const C zc = slots[k * NL + l], zp = slots[((N - k) % N) * NL + (l ^ 1)], pv = pk[j];
      C pp{0.f, 0.f};
      if (mb != 0.f) pp = ld2(p + (size_t)((N - row_y) % N) * NH + (size_t)((N - k) % N) * rowstride);
      C rv = rk[j];
      rv.x -= alpha * (ma * pv.x + mb * pp.x + (ca * zc.x + cb * zp.x));
      rv.y -= alpha * (ma * pv.y - mb * pp.y + (ca * zc.y - cb * zp.y));
      st2(r + base + (size_t)k * rowstride, rv);
      const float m2 = rv.x * rv.x + rv.y * rv.y, i0 = 1.f / (c0 * c0), iN = 1.f / (cN * cN);
      a_rr.add(m2);
      a_rc.add((i0 > iN ? i0 : iN) * m2);
    };
    if (mine) {
#pragma unroll
      for (int j = 0; j < R1; ++j) {
        const int k = t + j * N1;
        if (!AHEAD) ask(0, k);
        update(AHEAD ? j : 0, k);
      }
    }
  }
  const double s1 = block_sum_acc(a_rr, red);
  const double s2 = block_sum_acc(a_rc, red);
  if (tid == 0) {
    partials[0] = s1;
    partials[1] = s2;
  }
}

template <int N> WF_D size_t dslot(int kx, int ky, int kz);
// entry u (u = nh: k = 0) of r and, on the kz = 0 plane, its conjugate's
template <int N> WF_D void restore_entry(float2* r, const float2* rsave, const int4* modes, int nh, int u) {
  if (u == nh) {
    r[0] = rsave[2 * nh];
    return;
  }
  const int4 md = modes[u];
  r[dslot<N>(md.x, md.y, md.z)] = rsave[2 * u];
  if (md.z == 0) r[dslot<N>(-md.x, -md.y, 0)] = rsave[2 * u + 1];
}

// y pass: complex transform along y of every (x, kz) line, in place.  With fin.n1 > 0 the first row of CTAs takes alpha
// (YFin).  grid (N/2 / NL, N + (fin.n1 > 0), systems)
template <class G, int DIR>
__global__ void __launch_bounds__(G::NT, G::MINB)
k_ln_ypass(float2* __restrict__ T, const float2* __restrict__ twtab, CgScal* __restrict__ sc, Bat bt, YFin fin) {
  using C = cx<float>;
  constexpr int N = G::N, NH = G::NH, NL = G::NL, R1 = G::R1, N1 = G::N1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  C* slots = reinterpret_cast<C*>(smem_raw);
  float2* tw = reinterpret_cast<float2*>(slots + N * NL);
  const int z = blockIdx.z, tid = threadIdx.x, l = tid % NL, t = tid / NL;
  ln_load_tw<N>(tw, twtab, tid, G::NT);
  chain_start();
  if (sc && finished(sc + z)) return;
  int x = blockIdx.y;
  if constexpr (DIR < 0) {
    if (fin.n1 > 0 && x-- == 0) {
      if (blockIdx.x != 0) return;
      for (int u = tid; u <= fin.nh; u += G::NT)
        restore_entry<N>(fin.r + z * bt.spec, fin.rsave + (size_t)z * (2 * fin.nh + 1), fin.modes, fin.nh, u);
      fin_alpha(fin.part + (size_t)z * bt.part, fin.n1, fin.off, fin.n2, sc + z, reinterpret_cast<double*>(smem_raw));
      return;
    }
  }
  float2* p = T + z * bt.spec + (size_t)x * N * NH + blockIdx.x * NL + l;
  C v[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q) v[q] = ld2(p + (size_t)(q * N1 + t) * NH);
  __syncthreads();
  ln_forward<N, typename G::PL, DIR>(v, slots + l, ColMap<NL>{}, t, tw, [&](int k, C X, int) { st2(p + (size_t)k * NH, X); });
}

// ---- z passes: rows of N reals as H = N/2 complex elements; thread t of a row holds n1 (H / R1) + t -----------
// Rows are padded so that consecutive ones continue on the next banks (512^3: 0.48 ms with rows a multiple of 32
// banks apart).
template <int M> struct F32ZPlan { using T = typename F32Plan<M>::T; };
template <> struct F32ZPlan<72> { using T = LnRad<12, 6, 1>; };
template <> struct F32ZPlan<96> { using T = LnRad<12, 8, 1>; };
template <int N_, int TMAX, int MINB_ = 0, class PL_ = typename F32ZPlan<N_ / 2>::T> struct LZ {
  using PL = PL_;
  using C = cx<float>;
  static constexpr int N = N_, H = N / 2, R1 = PL::r1, N1 = H / R1, MINB = MINB_;
  static constexpr int NL = div_le(N * N, TMAX / N1);  // rows per CTA
  static constexpr int NT = NL * N1;
  static constexpr int SH = (PL::r3 > 1 ? PL::r3 : PL::r2) == 16 ? 4 : 3;
  using Map = PadMapT<SH>;
  static constexpr int LS = ln_padded(H, SH, N1, 16);
  static constexpr int GZ = N * N / NL;
  static constexpr size_t SMEM = (size_t)(NL * LS + N) * sizeof(C);
};
// packed X_k from the length-H transform Z, and Z_k from the packed X (slots in natural order; tw[k] =
// exp(-2 pi i k / N))
template <int N, class MAP> WF_D cx<float> ln_r2c(const cx<float>* s, const MAP& map, int k, const float2* tw) {
  constexpr int H = N / 2;
  const cx<float> a = s[map(k)];
  if (k == 0) return cx<float>{a.x + a.y, a.x - a.y};
  const cx<float> b = s[map(H - k)], d = ln_twid<-1>(cx<float>{a.x - b.x, a.y + b.y}, tw[k]);
  return cx<float>{0.5f * (a.x + b.x + d.y), 0.5f * (a.y - b.y - d.x)};
}
template <int N, class MAP> WF_D cx<float> ln_c2r(const cx<float>* s, const MAP& map, int k, const float2* tw) {
  constexpr int H = N / 2;
  const cx<float> a = s[map(k)];
  if (k == 0) return cx<float>{a.x + a.y, a.x - a.y};
  const cx<float> b = s[map(H - k)], d = ln_twid<+1>(cx<float>{a.x - b.x, a.y + b.y}, tw[k]);
  return cx<float>{a.x + b.x - d.y, a.y - b.y + d.x};
}

// The line's packed X in v (natural positions) -> real samples times D, transformed forward, in the line's slots in
// natural order (a barrier after it); the sum of D T^2 goes to acc.
template <class G>
WF_D void ln_turn(cx<float> (&v)[G::R1], cx<float>* s, int t, const float2* tw, const float2* __restrict__ d, AccF* acc) {
  using C = cx<float>;
  using Map = typename G::Map;
  constexpr int N = G::N, H = G::H, R1 = G::R1, N1 = G::N1;
  float2 dv[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q) s[Map{}(q * N1 + t)] = v[q];
#pragma unroll
  for (int q = 0; q < R1; ++q) dv[q] = __ldg(d + q * N1 + t);
  __syncthreads();
  ln_inverse<H, typename G::PL, +1, 2>(v, s, Map{}, t, tw, [&](int k) { return ln_c2r<N>(s, Map{}, k, tw); });
  float part = 0.f;
#pragma unroll
  for (int q = 0; q < R1; ++q) {
    const C T = v[q];
    v[q] = C{T.x * dv[q].x, T.y * dv[q].y};
    if (acc) {
      part += v[q].x * T.x + v[q].y * T.y;
      if (q % 2 == 1 || q == R1 - 1) {
        acc->add(part);
        part = 0.f;
      }
    }
  }
  __syncthreads();  // the inverse's last reads of the slots
  ln_forward_nat<H, typename G::PL, -1, 2>(v, s, Map{}, t, tw);
}

// z turn: each (x, y) line packed -> real, times D, -> packed; partial of D T^2.  grid (GZ, 1, systems)
template <class G>
__global__ void __launch_bounds__(G::NT, G::MINB)
k_ln_zturn(float2* __restrict__ spec, const float* __restrict__ D, const float2* __restrict__ twtab,
           double* __restrict__ partials, const CgScal* __restrict__ sc, Bat bt) {
  using C = cx<float>;
  using Map = typename G::Map;
  constexpr int N = G::N, H = G::H, R1 = G::R1, N1 = G::N1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  C* slots = reinterpret_cast<C*>(smem_raw);
  float2* tw = reinterpret_cast<float2*>(slots + G::NL * G::LS);
  __shared__ double red[32];
  const int z = blockIdx.z, tid = threadIdx.x, l = tid / N1, t = tid % N1;
  ln_load_tw<N>(tw, twtab, tid, G::NT);
  chain_start();
  if (sc && finished(sc + z)) return;
  const size_t row = (size_t)blockIdx.x * G::NL + l;
  float2* line = spec + z * bt.spec + row * H;
  C v[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q) v[q] = ld2(line + q * N1 + t);
  AccF acc;
  C* s = slots + l * G::LS;
  ln_turn<G>(v, s, t, tw, reinterpret_cast<const float2*>(D + z * bt.real) + row * H, &acc);
#pragma unroll
  for (int q = 0; q < R1; ++q) st2(line + q * N1 + t, ln_r2c<N>(s, Map{}, q * N1 + t, tw));
  const double sum = block_sum_acc(acc, red);
  if (tid == 0) partials[(size_t)z * bt.part + blockIdx.x] = sum;
}

// z stage of the coarse projection (the z turn without its full store): the kz = 0..K coefficients, element 0
// without the kz = N/2 plane packed beside it.  grid (GZ, 1, systems)
template <class G>
__global__ void __launch_bounds__(G::NT, G::MINB)
k_ln_zcoarse(const float2* __restrict__ spec, const float* __restrict__ D, const float2* __restrict__ twtab,
             float2* __restrict__ gz, int K, const CgScal* __restrict__ sc, Bat bt, size_t gzs) {
  using C = cx<float>;
  using Map = typename G::Map;
  constexpr int N = G::N, H = G::H, R1 = G::R1, N1 = G::N1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  C* slots = reinterpret_cast<C*>(smem_raw);
  float2* tw = reinterpret_cast<float2*>(slots + G::NL * G::LS);
  const int z = blockIdx.z, tid = threadIdx.x, l = tid / N1, t = tid % N1;
  ln_load_tw<N>(tw, twtab, tid, G::NT);
  chain_start();
  if (finished(sc + z)) return;
  const size_t row0 = (size_t)blockIdx.x * G::NL, row = row0 + l;
  const float2* line = spec + z * bt.spec + row * H;
  C v[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q) v[q] = ld2(line + q * N1 + t);
  ln_turn<G>(v, slots + l * G::LS, t, tw, reinterpret_cast<const float2*>(D + z * bt.real) + row * H, nullptr);
  gz += z * gzs + row0 * (K + 1);
  for (int e = tid; e < G::NL * (K + 1); e += G::NT) {
    const int ll = e / (K + 1), k = e % (K + 1);
    C X = ln_r2c<N>(slots + ll * G::LS, Map{}, k, tw);
    if (k == 0) X.y = 0.f;
    st2(gz + e, X);
  }
}

// ---- whole x-planes: the middle of an iteration in one kernel ---------------------------------------------------
// Up to 72 launches and their ramps bound an iteration.  Here one CTA holds a plane (N x N/2 complex) in shared memory: the
// inverse y transforms, the z turn and the forward y transforms move 3 spectra instead of 7 and are one launch
// instead of three, and the coarse stage (y, z, the DFT along y at the coarse modes) is one instead of three.
// A plane is stored as N padded rows; column and row lines work in place in it, with the same first radix along y
// and z, so that the thread grids agree.  Mixed solve at 64^3: 4.33 -> 4.08 ms.  Larger planes leave one CTA
// per SM, whose loads, transforms and stores do not overlap: 144^3 alone 8.80 -> 8.18 ms, but twelve systems of 64^3
// to 192^3 together 56.7 -> 63.5, and the choice may not depend on the company a system keeps (same bits in any batch).
template <int N> struct F32PlanePlan { using Y = LnRad<0, 0, 0>; using Z = LnRad<0, 0, 0>; };
#define WF_PLAN(M, A, B, C, D, E) \
  template <> struct F32PlanePlan<M> { using Y = LnRad<A, B, C>; using Z = LnRad<D, E, 1>; }
WF_PLAN(16, 4, 4, 1, 4, 2);
WF_PLAN(24, 4, 6, 1, 4, 3);
WF_PLAN(32, 4, 8, 1, 4, 4);
WF_PLAN(48, 6, 8, 1, 6, 4);
WF_PLAN(64, 8, 8, 1, 8, 4);
WF_PLAN(72, 6, 12, 1, 6, 6);
#undef WF_PLAN
constexpr int kPlaneMax = 72;
template <int N_> struct LP {
  using PY = typename F32PlanePlan<N_>::Y;
  using PZ = typename F32PlanePlan<N_>::Z;
  using Map = PadMapT<3>;
  static constexpr int N = N_, H = N / 2, R1 = PY::r1, NY = N / R1, NZ = H / R1;
  static constexpr int NT = H * NY, MINB = 768 / NT > 1 ? cmin(16, 768 / NT) : 1;
  static constexpr int LS = ln_padded(H, 3, NZ, 16);  // slots of a row
  static constexpr size_t SMEM = (size_t)(N * LS + N) * sizeof(cx<float>);
  static_assert(PZ::r1 == R1 && N * NZ == NT && NT <= 1024 && PY::r1 * PY::r2 * PY::r3 == N && R1 * PZ::r2 == H, "plan");
};
template <int LS> struct RowMap {
  WF_D int operator()(int p) const { return p * LS; }
};

// COARSE: T (read only) -> Gy[ky + K][kz][x], the DFT along y at |ky| <= K of the z turn's kz <= K (k_ycoarse's).
// Otherwise: T -> FFT_y FFT_z (D IFFT_z IFFT_y T) in place, the partial sum of D T^2, and the last CTA's alpha
// (YFin).  grid (N, 1, systems)
template <int N, bool COARSE>
__global__ void __launch_bounds__(LP<N>::NT, LP<N>::MINB)
k_ln_plane(float2* __restrict__ T, const float* __restrict__ D, const float2* __restrict__ twtab,
           double* __restrict__ partials, CgScal* __restrict__ sc, Bat bt, YFin fin, float2* __restrict__ gy, int K,
           size_t gys) {
  using C = cx<float>;
  using G = LP<N>;
  using Map = typename G::Map;
  constexpr int H = G::H, R1 = G::R1, NY = G::NY, NZ = G::NZ, LS = G::LS;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  C* plane = reinterpret_cast<C*>(smem_raw);
  float2* tw = reinterpret_cast<float2*>(plane + N * LS);
  __shared__ double red[32];
  const int z = blockIdx.z, tid = threadIdx.x, x = blockIdx.x;
  const int kz = tid % H, yt = tid / H, y = tid / NZ, zt = tid % NZ;  // column line and row line of the thread
  ln_load_tw<N>(tw, twtab, tid, G::NT);
  chain_start();
  if (sc && finished(sc + z)) return;
  float2* t = T + z * bt.spec + (size_t)x * N * H;
  C v[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q) v[q] = ld2(t + (size_t)(q * NY + yt) * H + kz);
  __syncthreads();  // twiddles
  ln_forward_nat<N, typename G::PY, +1, 1>(v, plane + Map{}(kz), RowMap<LS>{}, yt, tw);
  AccF acc;
  const float2* d = reinterpret_cast<const float2*>(D + z * bt.real) + ((size_t)x * N + y) * H;
  C* s = plane + y * LS;
  float2 dv[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q) dv[q] = __ldg(d + q * NZ + zt);
  ln_inverse<H, typename G::PZ, +1, 2>(v, s, Map{}, zt, tw, [&](int k) { return ln_c2r<N>(s, Map{}, k, tw); });
  float part = 0.f;
#pragma unroll
  for (int q = 0; q < R1; ++q) {
    const C r = v[q];
    v[q] = C{r.x * dv[q].x, r.y * dv[q].y};
    if constexpr (!COARSE) {
      part += v[q].x * r.x + v[q].y * r.y;
      if (q % 2 == 1 || q == R1 - 1) {
        acc.add(part);
        part = 0.f;
      }
    }
  }
  __syncthreads();  // the inverse's last reads of the slots
  ln_forward_nat<H, typename G::PZ, -1, 2>(v, s, Map{}, zt, tw);
  if constexpr (COARSE) {
    // kz <= K of every row (element 0 without the kz = N/2 plane), held by the row's first elements
    const int KZ = K + 1;
    constexpr int PER = (N * (kDeflMaxRadius + 1) + G::NT - 1) / G::NT;
    C keep[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int e = tid + i * G::NT;
      if (e < N * KZ) {
        keep[i] = ln_r2c<N>(plane + (e / KZ) * LS, Map{}, e % KZ, tw);
        if (e % KZ == 0) keep[i].y = 0.f;
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int e = tid + i * G::NT;
      if (e < N * KZ) plane[e] = keep[i];
    }
    __syncthreads();
    // four lanes per output, each over a quarter of the rows
    const int nout = (2 * K + 1) * KZ;
    gy += z * gys;
    for (int o4 = tid; o4 < (4 * nout + 31) / 32 * 32; o4 += G::NT) {
      const int o = o4 / 4, q4 = o4 % 4, ky = o / KZ - K, kc = o % KZ, step = (ky + N) % N;
      float sr = 0.f, si = 0.f;
      if (o < nout) {
        int e = (int)((unsigned)(q4 * (N / 4)) * (unsigned)step % N);
        for (int row = q4 * (N / 4); row < (q4 + 1) * (N / 4); ++row) {
          const C a = plane[row * KZ + kc];
          const float2 w = tw[e];
          sr += a.x * w.x - a.y * w.y;
          si += a.x * w.y + a.y * w.x;
          e += step;
          if (e >= N) e -= N;
        }
      }
      const unsigned m = __activemask();
      sr += __shfl_xor_sync(m, sr, 1);
      si += __shfl_xor_sync(m, si, 1);
      sr += __shfl_xor_sync(m, sr, 2);
      si += __shfl_xor_sync(m, si, 2);
      if (q4 == 0 && o < nout) gy[(size_t)o * N + x] = make_float2(sr, si);
    }
  } else {
#pragma unroll
    for (int q = 0; q < R1; ++q) v[q] = ln_r2c<N>(s, Map{}, q * NZ + zt, tw);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < R1; ++q) s[Map{}(q * NZ + zt)] = v[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < R1; ++q) v[q] = plane[(q * NY + yt) * LS + Map{}(kz)];
    __syncthreads();
    ln_forward<N, typename G::PY, -1>(v, plane + Map{}(kz), RowMap<LS>{}, yt, tw,
                                      [&](int k, C X, int) { st2(t + (size_t)k * H + kz, X); });
    const double sum = block_sum_acc(acc, red);
    partials += (size_t)z * bt.part;
    if (tid == 0) partials[fin.off + x] = sum;
    if (fin.n1 == 0 || !last_cta(&sc[z].tick[0], gridDim.x)) return;
    for (int u = tid; u <= fin.nh; u += G::NT)
      restore_entry<N>(fin.r + z * bt.spec, fin.rsave + (size_t)z * (2 * fin.nh + 1), fin.modes, fin.nh, u);
    fin_alpha(partials, fin.n1, fin.off, gridDim.x, sc + z, red);
  }
}

}  // namespace wf
