// wf_assign.cu -- supersampled mass assignment (Sec. 3.1.2 of Kitaura et al. 2009, Eq. def:ngrid).
//
// Step 1: each galaxy is placed on the fine grid (s n)^3 with CIC or TSC weights in fixed
//         point (Q16 per axis, product Q48) by 64-bit integer atomics, so the fine grid is
//         exact and independent of the order in which galaxies land.
// Step 2: the ideal discrete low-pass filter (keep modes with every |k_i| < n/2, drop the
//         coarse Nyquist planes) and sampling at n^3.  The filter is a box in k and therefore
//         separable.  Per axis, with the even and odd samples e_m, o_m of a line of 2n and
//         X_k = E_k + exp(-i pi k / n) O_k its low modes,
//           y_m = e_m - (-1)^m A / n + (1/n) sum_{|k| < n/2} exp(-i pi k / n) O_k exp(2 pi i k m / n),
//         A = sum (-1)^m e_m: the even samples without their Nyquist mode, plus the odd samples moved
//         by half a coarse cell.  Only the odd samples are transformed, and as the shift is a
//         real circulant, two lines go as the real and imaginary part of one complex line of n.
//         Three passes (z, y, x) each halve one axis: (2n)^3 -> (2n)^2 n -> 2n n^2 -> n^3.
#include "wf_ctx.h"
#include "wf_fix.cuh"
#include "wf_spectral.cuh"

namespace wf {

// ------------------------------------------------------------------------------------------
// step 1: fixed-point CIC / TSC atomics
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ int axis_nodes(double x, double scale, long long nf, int scheme,
                                          long long* node, unsigned long long* wt) {
  const double u = __dmul_rn(x, scale);
  if (!(fabs(u) < 4503599627370496.0)) return -1;  // 2^52: floor exact, non-finite rejected
  const long long m = nf * 65536LL;
  long long q = (long long)floor(u);
  q %= m;
  if (q < 0) q += m;
  if (scheme == WF_CIC) {
    const long long i = q >> 16;
    const unsigned long long f = (unsigned long long)(q & 0xFFFF);
    node[0] = i % nf;
    node[1] = (i + 1) % nf;
    wt[0] = 65536ULL - f;
    wt[1] = f;
    return 2;
  }
  const long long qp = q + 32768;
  const long long j = qp >> 16;
  const long long D = (qp & 0xFFFF) - 32768;  // offset from node j, [-2^15, 2^15)
  const unsigned long long a = (unsigned long long)(32768 - D), b = (unsigned long long)(32768 + D);
  const unsigned long long wm = (a * a) >> 17, wp = (b * b) >> 17;
  node[0] = ((j - 1) % nf + nf) % nf;
  node[1] = j % nf;
  node[2] = (j + 1) % nf;
  wt[0] = wm;
  wt[1] = 65536ULL - wm - wp;
  wt[2] = wp;
  return 3;
}

__global__ void __launch_bounds__(256)
k_assign(const double* __restrict__ pos, long long n_gal, long long nf, double scale, int scheme,
         unsigned long long* __restrict__ fine, int* __restrict__ err) {
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (g >= n_gal) return;
  long long nd[3][3];
  unsigned long long wt[3][3];
  int cnt = 0;
  for (int a = 0; a < 3; ++a) {
    cnt = axis_nodes(pos[3 * g + a], scale, nf, scheme, nd[a], wt[a]);
    if (cnt < 0) {
      atomicOr(err, 1);
      return;
    }
  }
  for (int i = 0; i < cnt; ++i)
    for (int j = 0; j < cnt; ++j) {
      const size_t rowb = ((size_t)nd[0][i] * nf + (size_t)nd[1][j]) * nf;
      const unsigned long long wij = wt[0][i] * wt[1][j];
      for (int k = 0; k < cnt; ++k) {
        const unsigned long long add = wij * wt[2][k];
        if (add == 0) continue;
        const unsigned long long old = atomicAdd(fine + rowb + nd[2][k], add);
        if (old + add < old) atomicOr(err, 2);
      }
    }
}

// Weighted assignment for the inverse-weighting estimator (Sec. 4, Eq. def:ngrid with galaxy
// mass wgt[g], e.g. 1 / w): each node contribution is the Q48 weight times wgt[g], rounded once
// to the nearest Q32 unit, so the grid is exact and independent of the order of the atomics.
__global__ void __launch_bounds__(256)
k_assign_weighted(const double* __restrict__ pos, const double* __restrict__ wgt, long long n_gal, long long nf,
                  double scale, int scheme, unsigned long long* __restrict__ fine, int* __restrict__ err) {
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (g >= n_gal) return;
  const double wg = wgt[g];
  if (!(wg >= 0.0) || !(wg < 4294967296.0)) {  // [0, 2^32): a contribution stays below 2^64
    atomicOr(err, 1);
    return;
  }
  long long nd[3][3];
  unsigned long long wt[3][3];
  int cnt = 0;
  for (int a = 0; a < 3; ++a) {
    cnt = axis_nodes(pos[3 * g + a], scale, nf, scheme, nd[a], wt[a]);
    if (cnt < 0) {
      atomicOr(err, 1);
      return;
    }
  }
  for (int i = 0; i < cnt; ++i)
    for (int j = 0; j < cnt; ++j) {
      const size_t rowb = ((size_t)nd[0][i] * nf + (size_t)nd[1][j]) * nf;
      const unsigned long long wij = wt[0][i] * wt[1][j];
      for (int k = 0; k < cnt; ++k) {
        const double q = __ull2double_rn(wij * wt[2][k]);  // exact: < 2^49
        const unsigned long long add = __double2ull_rn(__dmul_rn(__dmul_rn(q, wg), 1.0 / 65536.0));
        if (add == 0) continue;
        const unsigned long long old = atomicAdd(fine + rowb + nd[2][k], add);
        if (old + add < old) atomicOr(err, 2);
      }
    }
}

// fine grid in fixed-point units (2^-48 galaxies, 2^-32 weighted galaxies) -> FP64 counts
__global__ void k_q48_to_double(const unsigned long long* __restrict__ fine, double* __restrict__ out, size_t n,
                                double unit) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    out[i] = __ull2double_rn(fine[i]) * unit;
}

// ------------------------------------------------------------------------------------------
// step 2: one axis of the ideal low-pass, line pairs of 2N reals -> N reals, in 64-bit fixed point
// (wf_fix.cuh).  A pair's z_m = o_m(first) + i o_m(second) is transformed, multiplied by the half-sample
// shift (bin N/2: -A of the pair, so the inverse also subtracts the even samples' Nyquist mode) and
// transformed back; the even samples are added last, read again from L2 (a CTA's were read a few
// microseconds before) instead of being held in registers.  Between the two transforms the line is
// shifted right by fx_mid bits: the inverse's partial sums are below N ||(e, o)||_2, sqrt(N) times the
// forward's.  Units: with z scaled by 2^k, the result is 2^(k + a - fx_mid) y, a = floor(log2 N) from
// the shift table's factor 2^a / N.
// ------------------------------------------------------------------------------------------
constexpr int kNyqParts = 8;  // partial sums of A that the bin N/2 adds

// The multiplier between the transforms: bin k of the line (digits ph[k]); bin N/2 takes -A, the sum
// of the line's kNyqParts partial sums at ny[0], ny[st], ...
template <int N> struct LpShift {
  const int4* ph;
  const fxc* ny;
  int st;
  WF_D fxc operator()(int k, fxc X) const {
    if (k == N / 2) {
      fxc a{0, 0};
      for (int g = 0; g < kNyqParts; ++g) a = a + ny[g * st];
      X = fxc{-a.x, -a.y};
    }
    X = fxc{fx_rshift(X.x, fx_mid(N)), fx_rshift(X.y, fx_mid(N))};
    return fx_twid<-1>(X, __ldg(ph + k));
  }
};

template <bool A16> WF_D ulonglong2 ld_pair(const ulonglong2* p) {
  if constexpr (A16) return __ldg(p);
  const unsigned long long* q = reinterpret_cast<const unsigned long long*>(p);
  return make_ulonglong2(__ldg(q), __ldg(q + 1));
}

// z axis: rows of 2N integers (units of the grid) in pairs -> rows of N doubles.  Thread t of a pair
// holds elements n1 (N / R1) + t, so a warp reads and writes consecutive 16- and 8-byte pieces of a row.  Pairs
// of an all-zero CTA (most of the grid outside the survey) are written as zeros at once.  Bound by integer
// issue: 512^3 survey 32.0 ms (FP64 butterflies over all 2N samples) -> 3.52 ms (3.7 TB/s); asking for three
// CTAs per SM, where the compiler alone leaves two, took 3.96 to 3.52 (and nothing below 128).
template <int N> struct LpZ {
  static constexpr int R1 = fx_plan(N).r1, TPL = N / R1;
  static constexpr int NP = div_le(2 * N * N, TPL >= 128 ? 1 : 256 / TPL);  // pairs per CTA
  static constexpr int NT = NP * TPL;
  static constexpr int LS = ln_padded(N, 3, TPL, 8);
  static constexpr size_t SMEM = (size_t)(NP * LS + N + NP * (TPL + kNyqParts)) * 16;
};
// A16: the grid (a caller's fine_out) lies on a 16-byte boundary; otherwise its values are loaded one by one.
template <int N, bool A16>
__global__ void __launch_bounds__(LpZ<N>::NT, N >= 128 ? 3 : 0)
k_lowpass_z(const unsigned long long* __restrict__ in, double* __restrict__ out, double unit,
            const int4* __restrict__ twtab, const int4* __restrict__ phtab) {
  using G = LpZ<N>;
  constexpr int R1 = G::R1, N1 = N / R1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  fxc* slots = reinterpret_cast<fxc*>(smem_raw);
  int4* tw = reinterpret_cast<int4*>(slots + G::NP * G::LS);
  fxc* ny = reinterpret_cast<fxc*>(tw + N);  // per pair TPL thread sums, then kNyqParts partial sums
  __shared__ int s_len[G::NP];
  __shared__ unsigned s_q[G::NP];
  const int tid = threadIdx.x, l = tid / G::TPL, t = tid % G::TPL;
  const size_t row = 2 * ((size_t)blockIdx.x * G::NP + l);
  const ulonglong2* r0 = reinterpret_cast<const ulonglong2*>(in + row * (2 * N));
  const ulonglong2* r1 = r0 + N;
  ulonglong2 a[R1], b[R1];  // (even, odd) of both rows
  unsigned long long any = 0;
#pragma unroll
  for (int r = 0; r < R1; ++r) {
    a[r] = ld_pair<A16>(r0 + r * N1 + t);
    b[r] = ld_pair<A16>(r1 + r * N1 + t);
  }
#pragma unroll
  for (int r = 0; r < R1; ++r) any |= (a[r].x | a[r].y) | (b[r].x | b[r].y);
  if (tid < G::NP) {
    s_len[tid] = 0;
    s_q[tid] = 0;
  }
  if (!__syncthreads_or(any != 0)) {
    double* o = out + 2 * (size_t)blockIdx.x * G::NP * N;
    for (int e = tid; e < 2 * G::NP * N; e += G::NT) o[e] = 0.0;
    return;
  }
  fx_load_tw<N>(tw, twtab, tid, G::NT);
  if (any) atomicMax(&s_len[l], 64 - __clzll((long long)any));
  __syncthreads();
  const int len = s_len[l];  // every value of the pair is below 2^len
  {
    unsigned q = 0;
    auto top = [&](unsigned long long v) {  // v 2^(13 - len), rounded up
      const unsigned h = v ? (unsigned)(len > 13 ? v >> (len - 13) : v << (13 - len)) + 1u : 0u;
      q += h * h;  // 4 R1 <= 48 terms of at most 2^26
    };
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      top(a[r].x);
      top(a[r].y);
      top(b[r].x);
      top(b[r].y);
    }
    if (q) atomicAdd(&s_q[l], (q >> 7) + 1u);
  }
  __syncthreads();
  // sqrt(N) ||(e, o)|| 2^k <= 2^62
  const unsigned long long sq = (unsigned long long)s_q[l] * 128ull * (unsigned)N;
  const int k = len ? 62 + (13 - len) - ((64 - __clzll((long long)sq) + 1) >> 1) : 0;  // (0: a pair of zeros)
  auto fix = [&](unsigned long long v) { return (long long)(k >= 0 ? v << k : v >> -k); };
  fxc v[R1];
  {
    fxc e{0, 0};
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      const bool odd = (r * N1 + t) & 1;
      const long long ex = fix(a[r].x), ey = fix(b[r].x);
      e.x += odd ? -ex : ex;
      e.y += odd ? -ey : ey;
      v[r] = fxc{fix(a[r].y), fix(b[r].y)};
    }
    ny[l * G::TPL + t] = e;
  }
  __syncthreads();
  fxc* parts = ny + G::NP * G::TPL + l * kNyqParts;
  for (int g = t; g < kNyqParts; g += G::TPL) {
    fxc e{0, 0};
    for (int u = g; u < G::TPL; u += kNyqParts) e = e + ny[l * G::TPL + u];
    parts[g] = e;
  }
  ln_convolve<N, FxPlan<N>>(v, slots + l * G::LS, PadMap{}, t, tw, LpShift<N>{phtab, parts, 1});
  constexpr int A = fx_floor_log2(N) - fx_mid(N);
  const int ke = k + A;  // the even samples in the result's units
  auto fixe = [&](unsigned long long w) { return (long long)(ke >= 0 ? w << ke : w >> -ke); };
  const double c = unit * fx_pow2(-ke);
  double *o0 = out + row * N, *o1 = o0 + N;
#pragma unroll
  for (int r = 0; r < R1; ++r) {
    const int m = r * N1 + t;
    o0[m] = __ll2double_rn(fixe(__ldg(&r0[m].x)) + v[r].x) * c;
    o1[m] = __ll2double_rn(fixe(__ldg(&r1[m].x)) + v[r].y) * c;
  }
}

// y axis (AXIS 1, [2N][2N][N] -> [2N][N][N], fixed x = blockIdx.y) and x axis (AXIS 2, [2N][N][N] -> N^3, fixed
// y = blockIdx.y): the pairs are the double2 columns of consecutive z, NL of them per CTA.  512^3: y
// 26.1 -> 3.87 ms, x 13.1 -> 2.10 ms (1.6 TB/s; integer issue and the FP64 pipe's conversions share the
// time).  Four columns per CTA from 256 up: eight took 4.5 (y) and 2.3 ms, two 4.2 and 2.6.  Three CTAs per
// SM below 256 (216^3: y 0.34 -> 0.285 ms), which spilled to 4.08 ms at 512^3.
template <int N> struct LpC {
  static constexpr int R1 = fx_plan(N).r1, TPL = N / R1;
  static constexpr int NL = div_le(N / 2, N >= 256 ? 4 : 8);
  static constexpr int NT = NL * TPL;
  static constexpr size_t SMEM = (size_t)(N * NL + N + NL * (TPL + kNyqParts)) * 16;
};
// A16: the output (AXIS 2: a caller's n_obs) lies on a 16-byte boundary.
template <int N, int AXIS, bool A16>
__global__ void __launch_bounds__(LpC<N>::NT, N >= 128 && N < 256 ? 3 : 0)
k_lowpass_c(const double* __restrict__ in, double* __restrict__ out, const int4* __restrict__ twtab,
            const int4* __restrict__ phtab) {
  using G = LpC<N>;
  constexpr int R1 = G::R1, N1 = N / R1, NL = G::NL;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  fxc* slots = reinterpret_cast<fxc*>(smem_raw);
  int4* tw = reinterpret_cast<int4*>(slots + N * NL);
  double2* pa = reinterpret_cast<double2*>(tw + N);       // TPL thread sums per column
  fxc* parts = reinterpret_cast<fxc*>(pa + NL * G::TPL);  // kNyqParts partial sums per column
  __shared__ int s_e[NL];
  __shared__ unsigned s_q[NL];
  const int tid = threadIdx.x, l = tid % NL, t = tid / NL;
  const size_t stride = AXIS == 1 ? N : (size_t)N * N;  // of the line, in doubles
  const size_t first = (AXIS == 1 ? (size_t)blockIdx.y * 2 * N * N : (size_t)blockIdx.y * N) + 2 * ((size_t)blockIdx.x * NL + l);
  const double* src = in + first;
  double2 e[R1], o[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r) {
    const size_t m = r * N1 + t;
    e[r] = __ldg(reinterpret_cast<const double2*>(src + (2 * m) * stride));
    o[r] = __ldg(reinterpret_cast<const double2*>(src + (2 * m + 1) * stride));
  }
  if (tid < NL) {
    s_e[tid] = FxScale::kMin;
    s_q[tid] = 0;
  }
  fx_load_tw<N>(tw, twtab, tid, G::NT);
  __syncthreads();
  {
    int mx = 0;
    double2 s = make_double2(0.0, 0.0);
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      mx = max(max(mx, max(fx_exp(e[r].x), fx_exp(e[r].y))), max(fx_exp(o[r].x), fx_exp(o[r].y)));
      const bool odd = (r * N1 + t) & 1;
      s.x += odd ? -e[r].x : e[r].x;
      s.y += odd ? -e[r].y : e[r].y;
    }
    pa[t * NL + l] = s;
    if (mx > FxScale::kMin) atomicMax(&s_e[l], mx);
  }
  __syncthreads();
  const int emax = s_e[l];
  {
    unsigned q = 0;
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      const unsigned h0 = fx_top(e[r].x, emax), h1 = fx_top(e[r].y, emax);
      const unsigned h2 = fx_top(o[r].x, emax), h3 = fx_top(o[r].y, emax);
      q += h0 * h0 + h1 * h1;  // 4 R1 <= 48 terms of at most 2^26
      q += h2 * h2 + h3 * h3;
    }
    if (q) atomicAdd(&s_q[l], (q >> 7) + 1u);
  }
  __syncthreads();
  const int k = fx_scale(emax, s_q[l] + 1u, N);
  for (int g = t; g < kNyqParts; g += G::TPL) {
    double2 s = make_double2(0.0, 0.0);
    for (int u = g; u < G::TPL; u += kNyqParts) {
      s.x += pa[u * NL + l].x;
      s.y += pa[u * NL + l].y;
    }
    parts[g * NL + l] = fxc{fx_from(s.x, k), fx_from(s.y, k)};
  }
  fxc v[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r) v[r] = fxc{fx_from(o[r].x, k), fx_from(o[r].y, k)};
  ln_convolve<N, FxPlan<N>>(v, slots + l, ColMap<NL>{}, t, tw, LpShift<N>{phtab, parts + l, NL});
  constexpr int A = fx_floor_log2(N) - fx_mid(N);
  const double c = emax == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll) : fx_pow2(-(k + A));
  const size_t ostride = AXIS == 1 ? N : (size_t)N * N;
  double* dst = out + (AXIS == 1 ? (size_t)blockIdx.y * N * N : (size_t)blockIdx.y * N) + 2 * ((size_t)blockIdx.x * NL + l);
#pragma unroll
  for (int r = 0; r < R1; ++r) {
    const size_t m = r * N1 + t;
    const double2 ev = __ldg(reinterpret_cast<const double2*>(src + (2 * m) * stride));
    const double2 y = make_double2(fma(__ll2double_rn(v[r].x), c, ev.x), fma(__ll2double_rn(v[r].y), c, ev.y));
    if constexpr (A16) {
      *reinterpret_cast<double2*>(dst + m * ostride) = y;
    } else {
      dst[m * ostride] = y.x;
      dst[m * ostride + 1] = y.y;
    }
  }
}

template <class K>
static cudaError_t smem_attr(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int N>
static wf_status lowpass_sized(Ctx& c, const unsigned long long* fine, double* n_obs, double unit,
                               cudaStream_t st) {
  using Z = LpZ<N>;
  using C = LpC<N>;
  static_assert(2 * N * N % Z::NP == 0 && N / 2 % C::NL == 0 && Z::SMEM <= 227 * 1024 && C::SMEM <= 227 * 1024,
                "whole tiles");
  WF_TRY(c.fix_tables(N));
  const int4 *tw = c.fixed(N), *half = c.fixed_half(N);
  double *t1, *t2;
  WF_TRY(c.get("lp_t1", (size_t)4 * N * N * N * sizeof(double), (void**)&t1));
  WF_TRY(c.get("lp_t2", (size_t)2 * N * N * N * sizeof(double), (void**)&t2));
  auto kz = (uintptr_t)fine % 16 == 0 ? k_lowpass_z<N, true> : k_lowpass_z<N, false>;
  auto ky = k_lowpass_c<N, 1, true>;
  auto kx = (uintptr_t)n_obs % 16 == 0 ? k_lowpass_c<N, 2, true> : k_lowpass_c<N, 2, false>;
  WF_CUDA(smem_attr(kz, Z::SMEM));
  WF_CUDA(smem_attr(ky, C::SMEM));
  WF_CUDA(smem_attr(kx, C::SMEM));
  const double V = (double)N * N * N;
  c.launch("lowpass_z", 8 * (8 * V + 4 * V), st,
           [&] { kz<<<2 * N * N / Z::NP, Z::NT, Z::SMEM, st>>>(fine, t1, unit, tw, half); });
  WF_CUDA(cudaGetLastError());
  c.launch("lowpass_y", 8 * (4 * V + 2 * V), st,
           [&] { ky<<<dim3(N / 2 / C::NL, 2 * N), C::NT, C::SMEM, st>>>(t1, t2, tw, half); });
  WF_CUDA(cudaGetLastError());
  c.launch("lowpass_x", 8 * (2 * V + V), st,
           [&] { kx<<<dim3(N / 2 / C::NL, N), C::NT, C::SMEM, st>>>(t2, n_obs, tw, half); });
  WF_CUDA(cudaGetLastError());
  return WF_OK;
}

static wf_status assign_any(Ctx& c, const wf_grid& g, int scheme, const double* pos, const double* wgt,
                            int64_t n_gal, uint64_t* fine_out, double* n_obs, cudaStream_t st);

wf_status assign_run(Ctx& c, const wf_grid& g, int scheme, const double* pos, int64_t n_gal,
                     uint64_t* fine_out, double* n_obs, cudaStream_t st) {
  return assign_any(c, g, scheme, pos, nullptr, n_gal, fine_out, n_obs, st);
}

wf_status assign_weighted_run(Ctx& c, const wf_grid& g, int scheme, const double* pos, const double* wgt,
                              int64_t n_gal, uint64_t* fine_out, double* n_obs, cudaStream_t st) {
  if (n_gal > 0 && !wgt) return WF_ERR_ARG;
  return assign_any(c, g, scheme, pos, wgt, n_gal, fine_out, n_obs, st);
}

// wgt == nullptr: unit masses in Q48; else masses wgt[g] in Q32.
static wf_status assign_any(Ctx& c, const wf_grid& g, int scheme, const double* pos, const double* wgt,
                            int64_t n_gal, uint64_t* fine_out, double* n_obs, cudaStream_t st) {
  const int n = g.n, ss = g.supersample;
  if (!supported_size(n)) return WF_ERR_UNSUPPORTED;
  if (!(g.box > 0.0) || !(g.box < 1e300) || (ss != 1 && ss != 2) || (scheme != WF_CIC && scheme != WF_TSC) ||
      n_gal < 0 || (n_gal > 0 && !pos) || !n_obs)
    return WF_ERR_ARG;
  const long long nf = (long long)ss * n;
  const size_t nfine = (size_t)nf * nf * nf;
  unsigned long long* fine = reinterpret_cast<unsigned long long*>(fine_out);
  if (!fine) WF_TRY(c.get("fine", nfine * sizeof(uint64_t), (void**)&fine));
  int* err;
  WF_TRY(c.get("assign_err", 64, (void**)&err));
  WF_CUDA(cudaMemsetAsync(err, 0, sizeof(int), st));
  WF_CUDA(cudaMemsetAsync(fine, 0, nfine * sizeof(uint64_t), st));  // counted as a launch below
  c.prof.launches += 1;
  const double scale = ((double)nf * 65536.0) / g.box;
  const double unit = wgt ? 2.3283064365386963e-10 /* 2^-32 */ : 3.5527136788005009e-15 /* 2^-48 */;
  if (n_gal > 0) {
    c.launch("assign", 24.0 * n_gal + 16.0 * 27 * n_gal, st, [&] {
      if (wgt)
        k_assign_weighted<<<(unsigned)((n_gal + 255) / 256), 256, 0, st>>>(pos, wgt, (long long)n_gal, nf, scale,
                                                                           scheme, fine, err);
      else
        k_assign<<<(unsigned)((n_gal + 255) / 256), 256, 0, st>>>(pos, (long long)n_gal, nf, scale, scheme, fine, err);
    });
    WF_CUDA(cudaGetLastError());
  }
  if (ss == 1) {
    c.launch("q48", 16.0 * nfine, st, [&] { k_q48_to_double<<<1216, 256, 0, st>>>(fine, n_obs, nfine, unit); });
    WF_CUDA(cudaGetLastError());
  } else {
    wf_status s = WF_ERR_UNSUPPORTED;
    switch (n) {
#define WF_CASE(N) \
  case N:          \
    s = lowpass_sized<N>(c, fine, n_obs, unit, st); \
    break;
      WF_SIZES(WF_CASE)
#undef WF_CASE
    }
    if (s != WF_OK) return s;
  }
  int* h = reinterpret_cast<int*>(c.host_pinned);
  WF_CUDA(cudaMemcpyAsync(h, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  WF_CUDA(cudaStreamSynchronize(st));
  if (h[0] & 1) return WF_ERR_ARG;
  if (h[0] & 2) return WF_ERR_OVERFLOW;
  return WF_OK;
}

}  // namespace wf
