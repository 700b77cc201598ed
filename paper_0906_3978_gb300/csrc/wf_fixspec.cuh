// wf_fixspec.cuh -- the FP64 spectral passes (packed half spectra of wf_spectral.cuh, FP64 storage) with their
// transforms in 64-bit fixed point (wf_fix.cuh).  A CTA's threads load their elements straight into
// registers, the transform exchanges them through shared memory between its two or three passes, and the
// results go straight back: columns of the x and y passes as rows of 64 or 128 bytes, the rows of the
// z passes as consecutive 16-byte elements.  Bound by the FP64 pipe's conversions (four per complex element,
// more with an epilogue) beside the integer pipe; the FP64 butterflies they replace were bound by the
// FP64 pipe alone.  512^3 per launch, before -> after: y pass 3.53 -> 0.65 ms (3.3 TB/s), x multiplier 7.80 -> 1.26,
// z forward 4.48 -> 0.85, z inverse with the residual 5.52 -> 2.05.  Relative error of a smoothed field against
// long double: 3.4e-16 .. 6.6e-16 -> 1.2e-16 .. 2.1e-16 (32^3 .. 128^3).
#pragma once
#include "wf_fix.cuh"
#include "wf_spectral.cuh"

namespace wf {

// Geometry of the x / y passes: NL consecutive kz columns by N rows, one thread per line and element
// class mod N / R1.
template <int N> struct FxC {
  static constexpr int NH = N / 2;
  static constexpr int R1 = fx_plan(N).r1, N1 = N / R1;
  // up to 256 threads, but at small sizes eight columns, so that N (N/2) / NL CTAs cover the chip
  static constexpr int NL = div_le(NH, N >= 96 ? 256 / N1 : 8);
  static constexpr int NT = NL * N1;
  static constexpr int KB = NH / NL;  // column blocks per plane
  static constexpr size_t SMEM = (size_t)(N * NL + N) * 16;
  static_assert(NL >= 2, "a packed-column pair takes two line slots");
};

// y pass: complex transform along y of every (x, kz) line, in place.  With fin.n1 > 0 the first row of CTAs takes alpha
// (YFin).  S: the lines' range.  grid (N/2 / NL, N + (fin.n1 > 0), systems)
template <int N, int DIR, class S>
__global__ void __launch_bounds__(FxC<N>::NT)
k_fx_ypass(double2* __restrict__ T, const int4* __restrict__ twtab, CgScal* __restrict__ sc, Bat bt, YFin fin) {
  using G = FxC<N>;
  constexpr int R1 = G::R1, N1 = G::N1, NL = G::NL, NH = G::NH;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  fxc* slots = reinterpret_cast<fxc*>(smem_raw);
  int4* tw = reinterpret_cast<int4*>(slots + N * NL);
  __shared__ int se[NL];
  __shared__ unsigned sq[NL];
  const int z = blockIdx.z, tid = threadIdx.x, l = tid % NL, t = tid / NL;
  fx_load_tw<N>(tw, twtab, tid, G::NT);
  chain_start();
  if (sc && finished(sc + z)) return;
  int x = blockIdx.y;
  if constexpr (DIR < 0) {
    if (fin.n1 > 0 && x-- == 0) {
      if (blockIdx.x == 0)
        fin_alpha(fin.part + (size_t)z * bt.part, fin.n1, fin.off, fin.n2, sc + z, reinterpret_cast<double*>(smem_raw));
      return;
    }
  }
  double2* p = T + z * bt.spec + (size_t)x * N * NH + blockIdx.x * NL + l;
  double2 raw[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r) raw[r] = p[(size_t)(r * N1 + t) * NH];
  if (tid < NL) {
    se[tid] = S::kMin;
    sq[tid] = 0;
  }
  __syncthreads();
  const S f = fx_line_scale<S>(raw, &se[l], &sq[l], N);
  fxc v[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r) v[r] = fx_from2(raw[r], f);
  ln_forward<N, FxPlan<N>, DIR>(v, slots + l, ColMap<NL>{}, t, tw, [&](int k, fxc X, int) { p[(size_t)k * NH] = fx_to2(X, f); });
}

// tab[n2] = exp(-(kf r_s)^2 n2 / 2), the argument rounded operation by operation in the definition's order
static __global__ void k_gauss_table(double* __restrict__ tab, int n, double kf, double r_s) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  const double h = __dmul_rn(__dmul_rn(__dmul_rn(-0.5, kf), kf), (double)i);
  tab[i] = exp(__dmul_rn(__dmul_rn(h, r_s), r_s));
}

// ---- Fourier tables as Q62 digits ----------------------------------------------------------------
// tab[i] 2^-e as digits (high, low), in place; |tab[i]| < 2^e, e = exps[z estride].  One exponent serves a table, so
// an entry below 2^-9 of the largest has fewer bits than its FP64 value: the error of a product stays below
// 2^-62 max|tab| of the line's norm, where the transforms' FP64 storage leaves 2^-53 of it times the largest
// entry.  exps[] = kFxNanTab: a table with an infinity or NaN, whose every product is a NaN.  grid (., systems)
static __global__ void k_table_digits(double* __restrict__ tab, int len, const int* __restrict__ exps, int estride) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= len) return;
  tab += (size_t)blockIdx.y * len;
  long long q = __double2ll_rn(fx_scaled(tab[i], 62 - exps[blockIdx.y * estride]));
  const int l = (int)q;
  reinterpret_cast<int2*>(tab)[i] = make_int2((int)((q - l) >> 32), l);
}
WF_D fxc fx_scaleq(fxc a, int2 w) { return fxc{fx_mulq(a.x, w.x, w.y), fx_mulq(a.y, w.x, w.y)}; }
// (a + s b) / 2 of two digit pairs
WF_D int2 fx_mean(int2 a, int2 b, int s) {
  const long long x = ((long long)a.x << 32) + a.y, y = ((long long)b.x << 32) + b.y;
  const long long q = (x + s * y) >> 1;
  const int l = (int)q;
  return make_int2((int)((q - l) >> 32), l);
}

// x pass of a Fourier multiplier:  out = IFFT_x( tab (.) FFT_x(in) ), in != out.  The table holds digits
// with the system's power of two exps[z estride].  The packed column's multiplier pairs a line with the one at
// -ky: CTAs with blockIdx.x = N/2 / NL take both lines of a pair (ky <= N/2), the others skip column 0.
// grid (N/2 / NL + 1, N, systems)
template <int N> constexpr size_t fx_xmul_smem() { return FxC<N>::SMEM + (size_t)2 * N * 16; }
template <int N>
__global__ void __launch_bounds__(FxC<N>::NT)
k_fx_xmul(const double2* __restrict__ in, double2* __restrict__ out, const int2* __restrict__ tab,
          const int* __restrict__ exps, int estride, const int4* __restrict__ twtab, Bat bt) {
  using G = FxC<N>;
  constexpr int R1 = G::R1, N1 = G::N1, NL = G::NL, NH = G::NH;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  fxc* slots = reinterpret_cast<fxc*>(smem_raw);
  int4* tw = reinterpret_cast<int4*>(slots + N * NL);
  __shared__ int se[NL];
  __shared__ unsigned sq[NL];
  const int z = blockIdx.z, tid = threadIdx.x, l = tid % NL, t = tid / NL;
  const bool pair = blockIdx.x == G::KB;
  const int ky = blockIdx.y;
  if (pair && ky > N / 2) return;
  in += z * bt.spec;
  out += z * bt.spec;
  tab += z * bt.tab;
  const int ky_s = sfreq(ky, N);
  const size_t rowstride = (size_t)N * NH;
  // a pair's line slots 0 and 1 hold column 0 at ky and -ky, its other slots nothing
  const int row_y = pair && l == 1 ? (N - ky) % N : ky;
  const bool live = !pair || l < 2;
  const size_t base = (size_t)row_y * NH + (pair ? 0 : blockIdx.x * NL + l);
  double2 raw[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r)
    raw[r] = live ? __ldg(in + base + (size_t)(r * N1 + t) * rowstride) : make_double2(0.0, 0.0);
  if (tid < NL) {
    se[tid] = FxWide::kMin;
    sq[tid] = 0;
  }
  fx_load_tw<N>(tw, twtab, tid, G::NT);
  __syncthreads();
  const int ls = pair && l < 2 ? 0 : l;  // the two lines of a pair share a scale
  FxWide f = fx_line_scale<FxWide>(raw, &se[ls], &sq[ls], N);
  fxc v[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r) v[r] = fx_from2(raw[r], f);
  constexpr int H2 = fx_mid(N);
  const int te = exps[z * estride], sh = -(H2 + te);
  if (te == kFxNanTab) f.nan = 0x7ff80000u;
  if (!pair) {
    const int kz = blockIdx.x * NL + l, k0 = ky_s * ky_s + kz * kz;
    ln_convolve<N, FxPlan<N>>(v, slots + l, ColMap<NL>{}, t, tw, [&](int k, fxc X) {
      const int kxs = sfreq(k, N);
      return fx_scaleq(fxc{fx_rshift(X.x, H2), fx_rshift(X.y, H2)}, __ldg(tab + kxs * kxs + k0));
    });
    if (kz == 0) return;  // the packed column's pair CTA writes it
  } else {
    fxc* nat = reinterpret_cast<fxc*>(tw + N);  // both lines' spectra in natural order
    ln_forward<N, FxPlan<N>, -1>(v, slots + l, ColMap<NL>{}, t, tw, [&](int k, fxc X, int) {
      if (l < 2) nat[l * N + k] = fxc{fx_rshift(X.x, H2), fx_rshift(X.y, H2)};
    });
    __syncthreads();
    ln_inverse<N, FxPlan<N>, +1>(v, slots + l, ColMap<NL>{}, t, tw, [&](int k) {
      if (l >= 2) return fxc{0, 0};
      const int kxs = sfreq(k, N), n2 = kxs * kxs + ky_s * ky_s;
      const int2 m0 = __ldg(tab + n2), mN = __ldg(tab + n2 + NH * NH);
      const fxc a = fx_scaleq(nat[l * N + k], fx_mean(m0, mN, 1));
      const fxc b = fx_scaleq(nat[(1 - l) * N + (N - k) % N], fx_mean(m0, mN, -1));
      return fxc{a.x + b.x, a.y - b.y};  // m+ Z(k) + m- conj Z(-k)
    });
    if (l >= 2 || (l == 1 && row_y == ky)) return;
  }
#pragma unroll
  for (int r = 0; r < R1; ++r) out[base + (size_t)(r * N1 + t) * rowstride] = fx_to2(v[r], f, sh);
}

// x pass of the CG start:  out = tab (.) FFT_x(in),  partial of wgt |out|^2 (wgt 1 on column 0, 2 elsewhere)
// per CTA; FP64 table.  CTAs as in k_fx_xmul.
template <int N>
__global__ void __launch_bounds__(FxC<N>::NT)
k_fx_xfwd(const double2* __restrict__ in, double2* __restrict__ out, const double* __restrict__ tab,
          const int4* __restrict__ twtab, double* __restrict__ partials, Bat bt) {
  using G = FxC<N>;
  constexpr int R1 = G::R1, N1 = G::N1, NL = G::NL, NH = G::NH;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  fxc* slots = reinterpret_cast<fxc*>(smem_raw);
  int4* tw = reinterpret_cast<int4*>(slots + N * NL);
  __shared__ int se[NL];
  __shared__ unsigned sq[NL];
  __shared__ double red[32];
  const int z = blockIdx.z, tid = threadIdx.x, l = tid % NL, t = tid / NL;
  const bool pair = blockIdx.x == G::KB;
  const int ky = blockIdx.y;
  partials += (size_t)z * bt.part + blockIdx.y * gridDim.x + blockIdx.x;
  if (pair && ky > N / 2) {
    if (tid == 0) *partials = 0.0;
    return;
  }
  in += z * bt.spec;
  out += z * bt.spec;
  tab += z * bt.tab;
  const int ky_s = sfreq(ky, N);
  const size_t rowstride = (size_t)N * NH;
  const int row_y = pair && l == 1 ? (N - ky) % N : ky;
  const bool live = !pair || l < 2;
  const size_t base = (size_t)row_y * NH + (pair ? 0 : blockIdx.x * NL + l);
  double2 raw[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r)
    raw[r] = live ? __ldg(in + base + (size_t)(r * N1 + t) * rowstride) : make_double2(0.0, 0.0);
  if (tid < NL) {
    se[tid] = FxScale::kMin;
    sq[tid] = 0;
  }
  fx_load_tw<N>(tw, twtab, tid, G::NT);
  __syncthreads();
  const int ls = pair && l < 2 ? 0 : l;
  const FxScale f = fx_line_scale<FxScale>(raw, &se[ls], &sq[ls], N);
  fxc v[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r) v[r] = fx_from2(raw[r], f);
  AccD acc;
  if (!pair) {
    const int kz = blockIdx.x * NL + l, k0 = ky_s * ky_s + kz * kz;
    ln_forward<N, FxPlan<N>, -1>(v, slots + l, ColMap<NL>{}, t, tw, [&](int k, fxc X, int) {
      if (kz == 0) return;
      const int kxs = sfreq(k, N);
      const double m = __ldg(tab + kxs * kxs + k0);
      const double2 d = fx_to2(X, f), o = make_double2(d.x * m, d.y * m);
      out[base + (size_t)k * rowstride] = o;
      acc.add_prod(2.0 * o.x, o.x);
      acc.add_prod(2.0 * o.y, o.y);
    });
  } else {
    fxc* nat = reinterpret_cast<fxc*>(tw + N);
    ln_forward<N, FxPlan<N>, -1>(v, slots + l, ColMap<NL>{}, t, tw, [&](int k, fxc X, int) {
      if (l < 2) nat[l * N + k] = X;
    });
    __syncthreads();
    if (l < 2 && !(l == 1 && row_y == ky))
      for (int k = t; k < N; k += N1) {
        const int kxs = sfreq(k, N), n2 = kxs * kxs + ky_s * ky_s;
        const double m0 = __ldg(tab + n2), mN = __ldg(tab + n2 + NH * NH);
        const double a = 0.5 * (m0 + mN), b = 0.5 * (m0 - mN);
        const double2 zc = fx_to2(nat[l * N + k], f), zp = fx_to2(nat[(1 - l) * N + (N - k) % N], f);
        const double2 o = make_double2(a * zc.x + b * zp.x, a * zc.y - b * zp.y);
        out[base + (size_t)k * rowstride] = o;
        acc.add_prod(o.x, o.x);
        acc.add_prod(o.y, o.y);
      }
  }
  const double s = block_sum(acc.get(), red);
  if (tid == 0) *partials = s;
}

// x pass of s = C x:  out = IFFT_x( tab (.) in ), in != out; FP64 table.  grid (N/2 / NL, N, systems)
template <int N>
__global__ void __launch_bounds__(FxC<N>::NT)
k_fx_xinv(const double2* __restrict__ in, double2* __restrict__ out, const double* __restrict__ tab,
          const int4* __restrict__ twtab, Bat bt) {
  using G = FxC<N>;
  constexpr int R1 = G::R1, N1 = G::N1, NL = G::NL, NH = G::NH;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  fxc* slots = reinterpret_cast<fxc*>(smem_raw);
  int4* tw = reinterpret_cast<int4*>(slots + N * NL);
  __shared__ int se[NL];
  __shared__ unsigned sq[NL];
  const int z = blockIdx.z, tid = threadIdx.x, l = tid % NL, t = tid / NL;
  in += z * bt.spec;
  out += z * bt.spec;
  tab += z * bt.tab;
  const int ky = blockIdx.y, ky_s = sfreq(ky, N), kz = blockIdx.x * NL + l;
  const size_t rowstride = (size_t)N * NH, base = (size_t)ky * NH + kz;
  double2 raw[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r) {
    const int kx = r * N1 + t, kxs = sfreq(kx, N), n2 = kxs * kxs + ky_s * ky_s + kz * kz;
    const double2 c = __ldg(in + base + (size_t)kx * rowstride);
    const double m = __ldg(tab + n2);
    if (kz != 0) {
      raw[r] = make_double2(c.x * m, c.y * m);
    } else {
      const double mN = __ldg(tab + n2 + NH * NH), a = 0.5 * (m + mN), b = 0.5 * (m - mN);
      const double2 p = __ldg(in + (size_t)((N - ky) % N) * NH + (size_t)((N - kx) % N) * rowstride);
      raw[r] = make_double2(a * c.x + b * p.x, a * c.y - b * p.y);
    }
  }
  if (tid < NL) {
    se[tid] = FxScale::kMin;
    sq[tid] = 0;
  }
  fx_load_tw<N>(tw, twtab, tid, G::NT);
  __syncthreads();
  const FxScale f = fx_line_scale<FxScale>(raw, &se[l], &sq[l], N);
  fxc v[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r) v[r] = fx_from2(raw[r], f);
  ln_forward<N, FxPlan<N>, +1>(v, slots + l, ColMap<NL>{}, t, tw,
                    [&](int k, fxc X, int) { out[base + (size_t)k * rowstride] = fx_to2(X, f); });
}

// ---- z passes: rows of N reals as H = N/2 complex elements, thread t of a row holding n1 (H / R1) + t ----
template <int N> struct FxZ {
  static constexpr int H = N / 2, R1 = fx_plan(H).r1, N1 = H / R1;
  static constexpr int NL = div_le(N * N, 256 / N1);  // rows per CTA
  static constexpr int NT = NL * N1;
  static constexpr int LS = ln_padded(H, 3, N1, 8);
  static constexpr int GZ = N * N / NL;  // CTAs per system
  static constexpr size_t SMEM = (size_t)(NL * LS + N) * 16;
};

// X_k of the packed half spectrum from the length-H transform Z of x_2m + i x_2m+1 (slots in natural order)
template <int N, class MAP> WF_D fxc fx_r2c(const fxc* s, const MAP& map, int k, const int4* tw) {
  constexpr int H = N / 2;
  const fxc a = s[map(k)];
  if (k == 0) return fxc{a.x + a.y, a.x - a.y};
  const fxc b = s[map(H - k)];
  // halves first: X_k = (Z_k + conj Z_{H-k}) / 2 - (i/2) W_N^k (Z_k - conj Z_{H-k})
  const fxc ah{(a.x + 1) >> 1, (a.y + 1) >> 1}, bh{(b.x + 1) >> 1, (b.y + 1) >> 1};
  const fxc d = fx_twid<-1>(fxc{ah.x - bh.x, ah.y + bh.y}, tw[k]);
  return fxc{ah.x + bh.x + d.y, ah.y - bh.y - d.x};
}
// Z_k from the packed X: (X_k + conj X_{H-k}) + i W_N^-k (X_k - conj X_{H-k})
template <int N, class MAP> WF_D fxc fx_c2r(const fxc* s, const MAP& map, int k, const int4* tw) {
  constexpr int H = N / 2;
  const fxc a = s[map(k)];
  if (k == 0) return fxc{a.x + a.y, a.x - a.y};
  const fxc b = s[map(H - k)];
  const fxc d = fx_twid<+1>(fxc{a.x - b.x, a.y + b.y}, tw[k]);
  return fxc{a.x + b.x - d.y, a.y - b.y + d.x};
}
// The scale factor of a line's element count that bounds the C2R transform: with the packed X scaled by
// ||Z||_2 <= 2 sqrt(2) ||X||_2, its partial sums are below sqrt(8 H) ||X||_2.
template <int N> constexpr int fx_c2r_count() { return 8 * (N / 2); }

// z forward: real rows -> packed spectrum rows.  grid (GZ, 1, systems)
template <int N>
__global__ void __launch_bounds__(FxZ<N>::NT)
k_fx_zfwd(const double* __restrict__ in, double2* __restrict__ out, const int4* __restrict__ twtab,
          const CgScal* __restrict__ sc, Bat bt) {
  using G = FxZ<N>;
  constexpr int R1 = G::R1, N1 = G::N1, H = G::H;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  fxc* slots = reinterpret_cast<fxc*>(smem_raw);
  int4* tw = reinterpret_cast<int4*>(slots + G::NL * G::LS);  // exp(-2 pi i e / N)
  __shared__ int se[G::NL];
  __shared__ unsigned sq[G::NL];
  const int z = blockIdx.z, tid = threadIdx.x, l = tid / N1, t = tid % N1;
  if (sc && sc[z].done) return;
  const size_t row = (size_t)blockIdx.x * G::NL + l;
  const double2* src = reinterpret_cast<const double2*>(in + z * bt.real) + row * H;
  double2 raw[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r) raw[r] = __ldg(src + r * N1 + t);
  if (tid < G::NL) {
    se[tid] = FxWide::kMin;
    sq[tid] = 0;
  }
  fx_load_tw<N>(tw, twtab, tid, G::NT);
  __syncthreads();
  const FxWide f = fx_line_scale<FxWide>(raw, &se[l], &sq[l], H);
  fxc* s = slots + l * G::LS;
  fxc v[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r) v[r] = fx_from2(raw[r], f);
  ln_forward_nat<H, FxPlan<H>, -1, 2>(v, s, PadMap{}, t, tw);
  double2* dst = out + z * bt.spec + row * H;
  for (int k = t; k < H; k += N1) dst[k] = fx_to2(fx_r2c<N>(s, PadMap{}, k, tw), f);
}

// z inverse: packed spectrum rows -> real rows, value v = scl * C2R(in), then the modes of k_zinv
// (ZI_STORE out = v; ZI_RESID out = b - (v + nbar w s) with the partial sum of out^2).  grid (GZ, 1, systems)
template <int N, int MODE>
__global__ void __launch_bounds__(FxZ<N>::NT)
k_fx_zinv(const double2* __restrict__ in, double* __restrict__ out, const double* __restrict__ s,
          const double* __restrict__ w, const double* __restrict__ b, double scl, const int4* __restrict__ twtab,
          double* __restrict__ partials, const CgScal* __restrict__ sc, Bat bt) {
  using G = FxZ<N>;
  constexpr int R1 = G::R1, N1 = G::N1, H = G::H;
  static_assert(MODE == ZI_STORE || MODE == ZI_RESID, "mode");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  fxc* slots = reinterpret_cast<fxc*>(smem_raw);
  int4* tw = reinterpret_cast<int4*>(slots + G::NL * G::LS);
  __shared__ int se[G::NL];
  __shared__ unsigned sq[G::NL];
  __shared__ double red[32];
  const int z = blockIdx.z, tid = threadIdx.x, l = tid / N1, t = tid % N1;
  const double nbar = sc ? sc[z].nbar : 0.0;
  if (MODE != ZI_RESID && sc && sc[z].done == 4) return;
  const size_t row = (size_t)blockIdx.x * G::NL + l;
  const double2* src = in + z * bt.spec + row * H;
  double2 raw[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r) raw[r] = __ldg(src + r * N1 + t);
  if (tid < G::NL) {
    se[tid] = FxWide::kMin;
    sq[tid] = 0;
  }
  fx_load_tw<N>(tw, twtab, tid, G::NT);
  __syncthreads();
  const FxWide f = fx_line_scale<FxWide>(raw, &se[l], &sq[l], fx_c2r_count<N>());
  fxc* sl = slots + l * G::LS;
#pragma unroll
  for (int r = 0; r < R1; ++r) sl[PadMap{}(r * N1 + t)] = fx_from2(raw[r], f);
  __syncthreads();
  fxc v[R1];
  ln_inverse<H, FxPlan<H>, +1, 2>(v, sl, PadMap{}, t, tw, [&](int k) { return fx_c2r<N>(sl, PadMap{}, k, tw); });
  AccD acc;
  const size_t e0 = z * (bt.real / 2) + row * H;
#pragma unroll
  for (int r = 0; r < R1; ++r) {
    const size_t e = e0 + r * N1 + t;
    const double2 x = fx_to2(v[r], f);
    double2 val;
    if constexpr (MODE == ZI_RESID) {
      const double2 sv = __ldg(reinterpret_cast<const double2*>(s) + e);
      const double2 wv = __ldg(reinterpret_cast<const double2*>(w) + e);
      const double2 bv = __ldg(reinterpret_cast<const double2*>(b) + e);
      val.x = bv.x - (x.x * scl + nbar * wv.x * sv.x);
      val.y = bv.y - (x.y * scl + nbar * wv.y * sv.y);
      acc.add_prod(val.x, val.x);
      acc.add_prod(val.y, val.y);
    } else {
      val = make_double2(x.x * scl, x.y * scl);
    }
    reinterpret_cast<double2*>(out)[e] = val;
  }
  if constexpr (MODE == ZI_RESID) {
    const double sum = block_sum(acc.get(), red);
    if (tid == 0) partials[(size_t)z * bt.part + blockIdx.x] = sum;
  }
}

// ==========================================================================================
// The FP64 CG passes (the work of k_cg_xinv, k_cg_xupd and k_zturn): vector updates and sums in FP64,
// transforms in fixed point.  UNIT_M (every system preconditioned): m = 1 but at k = 0, where it is 0,
// and the m table holds 1 / c^2 instead, which the residual estimate would otherwise divide for.  108^3 per
// launch (events, with ~5 us of bracketing), FP64 butterflies -> here: x pass 1 58.8 -> 43 us, x pass 2 87 -> 43,
// z turn 103 -> 37, y pass 43 -> 16; the FP64 pipe's updates and conversions (about 55 per complex element and
// iteration) and the loads' latency at this size share the rest.  Each round's operands are requested
// before they are needed: with the loads between the stores, x pass 1 took 65 us.
// ==========================================================================================
template <bool UNIT_M> WF_D double cg_m(const double* mtab, int n2) {
  return UNIT_M ? (n2 == 0 ? 0.0 : 1.0) : __ldg(mtab + n2);
}
template <bool UNIT_M> WF_D double cg_ic2(const double* mtab, int n2, double c) {
  return UNIT_M ? __ldg(mtab + n2) : 1.0 / (c * c);
}

// x pass 1: p_new = r + beta p_old;  x += alpha_prev p_old;  T = IFFT_x(c (.) p_new);  partial of <p_new, m p_new>.
// The packed column takes its partner element from -ky in registers.  grid (N/2 / NL, N, systems)
template <int N, bool UNIT_M>
__global__ void __launch_bounds__(FxC<N>::NT)
k_fx_cg_xinv(const double2* __restrict__ r, double2* P0, double2* P1, double2* __restrict__ x, double2* __restrict__ T,
             const double* __restrict__ ctab, const double* __restrict__ mtab, const int4* __restrict__ twtab,
             double* __restrict__ partials, const CgScal* __restrict__ sc, Bat bt) {
  using G = FxC<N>;
  constexpr int R1 = G::R1, N1 = G::N1, NL = G::NL, NH = G::NH;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  fxc* slots = reinterpret_cast<fxc*>(smem_raw);
  int4* tw = reinterpret_cast<int4*>(slots + N * NL);
  __shared__ int se[NL];
  __shared__ unsigned sq[NL];
  __shared__ double red[32];
  const int z = blockIdx.z, tid = threadIdx.x, l = tid % NL, t = tid / NL;
  fx_load_tw<N>(tw, twtab, tid, G::NT);
  chain_start();
  sc += z;
  if (finished(sc)) return;
  const double2* __restrict__ pold = ((sc->lit & 1) ? P1 : P0) + z * bt.spec;
  double2* __restrict__ pnew = ((sc->lit & 1) ? P0 : P1) + z * bt.spec;
  r += z * bt.spec;
  x += z * bt.spec;
  T += z * bt.spec;
  ctab += z * bt.tab;
  mtab += z * bt.tab;
  const double beta = sc->beta, alpha = sc->alpha_prev;
  const int ky = blockIdx.y, ky_s = sfreq(ky, N), kz = blockIdx.x * NL + l;
  const size_t rowstride = (size_t)N * NH, base = (size_t)ky * NH + kz;
  double2 raw[R1];
  double acc = 0.0;  // half of the sum: the columns kz != 0 weigh 2
  constexpr int CH = R1 % 4 == 0 ? 4 : 3;  // elements whose loads are in flight together
  static_assert(R1 % CH == 0, "chunks");
#pragma unroll
  for (int q0 = 0; q0 < R1; q0 += CH) {
    double2 rv[CH], po[CH], xv[CH];
    double cv[CH];
#pragma unroll
    for (int j = 0; j < CH; ++j) {
      const int kx = (q0 + j) * N1 + t, kxs = sfreq(kx, N);
      const size_t e = base + (size_t)kx * rowstride;
      rv[j] = __ldg(r + e);
      po[j] = __ldg(pold + e);
      xv[j] = x[e];
      cv[j] = __ldg(ctab + kxs * kxs + ky_s * ky_s + kz * kz);
    }
#pragma unroll
    for (int j = 0; j < CH; ++j) {
      const int kx = (q0 + j) * N1 + t;
      const size_t e = base + (size_t)kx * rowstride;
      const double2 p = make_double2(rv[j].x + beta * po[j].x, rv[j].y + beta * po[j].y);
      pnew[e] = p;
      x[e] = make_double2(xv[j].x + alpha * po[j].x, xv[j].y + alpha * po[j].y);
      if (kz != 0) {
        if (UNIT_M) {
          acc = fma(p.x, p.x, fma(p.y, p.y, acc));
        } else {
          const int kxs = sfreq(kx, N);
          acc = fma(__ldg(mtab + kxs * kxs + ky_s * ky_s + kz * kz), p.x * p.x + p.y * p.y, acc);
        }
        raw[q0 + j] = make_double2(cv[j] * p.x, cv[j] * p.y);
      } else {
        raw[q0 + j] = p;  // raw for the pair below
      }
    }
  }
  if (kz == 0) {  // packed column: c and m act on the planes P0 = (Z + conj Z(-k)) / 2, PN = (Z - conj Z(-k)) / 2i
#pragma unroll
    for (int q0 = 0; q0 < R1; q0 += CH) {
      double2 rq[CH], pq[CH];
#pragma unroll
      for (int j = 0; j < CH; ++j) {
        const int kx = (q0 + j) * N1 + t;
        const size_t eq = (size_t)((N - ky) % N) * NH + (size_t)((N - kx) % N) * rowstride;
        rq[j] = __ldg(r + eq);
        pq[j] = __ldg(pold + eq);
      }
#pragma unroll
      for (int j = 0; j < CH; ++j) {
        const int kxs = sfreq((q0 + j) * N1 + t, N), n2 = kxs * kxs + ky_s * ky_s;
        const double2 p = raw[q0 + j];
        const double qx = rq[j].x + beta * pq[j].x, qy = rq[j].y + beta * pq[j].y;
        const double a0 = 0.5 * (p.x + qx), b0 = 0.5 * (p.y - qy), aN = 0.5 * (p.y + qy), bN = 0.5 * (qx - p.x);
        acc += 0.5 * (cg_m<UNIT_M>(mtab, n2) * (a0 * a0 + b0 * b0) + cg_m<UNIT_M>(mtab, n2 + NH * NH) * (aN * aN + bN * bN));
        const double c = __ldg(ctab + n2), cN = __ldg(ctab + n2 + NH * NH), a = 0.5 * (c + cN), b = 0.5 * (c - cN);
        raw[q0 + j] = make_double2(a * p.x + b * qx, a * p.y - b * qy);
      }
    }
  }
  if (tid < NL) {
    se[tid] = FxScale::kMin;
    sq[tid] = 0;
  }
  __syncthreads();
  const FxScale f = fx_line_scale<FxScale>(raw, &se[l], &sq[l], N);
  fxc v[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q) v[q] = fx_from2(raw[q], f);
  ln_forward<N, FxPlan<N>, +1>(v, slots + l, ColMap<NL>{}, t, tw,
                    [&](int k, fxc X, int) { T[base + (size_t)k * rowstride] = fx_to2(X, f); });
  const double sum = block_sum(2.0 * acc, red);
  if (tid == 0) partials[(size_t)z * bt.part + blockIdx.y * gridDim.x + blockIdx.x] = sum;
}

// x pass 2:  T^ = FFT_x(T);  q = m p + c T^;  r -= alpha q;  partials of <r, r> and an upper estimate of
// V_c ||C^-1 r||^2 (two per CTA).  CTAs as in k_fx_xmul.
template <int N, bool UNIT_M>
__global__ void __launch_bounds__(FxC<N>::NT)
k_fx_cg_xupd(const double2* __restrict__ T, double2* __restrict__ r, const double2* P0, const double2* P1,
             const double* __restrict__ ctab, const double* __restrict__ mtab, const int4* __restrict__ twtab,
             double* __restrict__ partials, const CgScal* __restrict__ sc, Bat bt) {
  using G = FxC<N>;
  constexpr int R1 = G::R1, N1 = G::N1, NL = G::NL, NH = G::NH;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  fxc* slots = reinterpret_cast<fxc*>(smem_raw);
  int4* tw = reinterpret_cast<int4*>(slots + N * NL);
  __shared__ int se[NL];
  __shared__ unsigned sq[NL];
  __shared__ double red[32];
  const int z = blockIdx.z, tid = threadIdx.x, l = tid % NL, t = tid / NL;
  fx_load_tw<N>(tw, twtab, tid, G::NT);
  chain_start();
  sc += z;
  if (finished(sc)) return;
  const bool pair = blockIdx.x == G::KB;
  const int ky = blockIdx.y;
  partials += (size_t)z * bt.part + 2 * (size_t)(blockIdx.y * gridDim.x + blockIdx.x);
  if (pair && ky > N / 2) {
    if (tid < 2) partials[tid] = 0.0;
    return;
  }
  const double2* __restrict__ p = ((sc->lit & 1) ? P0 : P1) + z * bt.spec;  // this iteration's p_new
  T += z * bt.spec;
  r += z * bt.spec;
  ctab += z * bt.tab;
  mtab += z * bt.tab;
  const double alpha = sc->alpha;
  const int ky_s = sfreq(ky, N);
  const size_t rowstride = (size_t)N * NH;
  const int row_y = pair && l == 1 ? (N - ky) % N : ky;
  const bool live = !pair || l < 2;
  const size_t base = (size_t)row_y * NH + (pair ? 0 : blockIdx.x * NL + l);
  double2 raw[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q)
    raw[q] = live ? __ldg(T + base + (size_t)(q * N1 + t) * rowstride) : make_double2(0.0, 0.0);
  if (tid < NL) {
    se[tid] = FxScale::kMin;
    sq[tid] = 0;
  }
  __syncthreads();
  const int ls = pair && l < 2 ? 0 : l;
  const FxScale f = fx_line_scale<FxScale>(raw, &se[ls], &sq[ls], N);
  fxc v[R1];
#pragma unroll
  for (int q = 0; q < R1; ++q) v[q] = fx_from2(raw[q], f);
  double rr = 0.0, rc = 0.0;
  if (!pair) {
    const int kz = blockIdx.x * NL + l, k0 = ky_s * ky_s + kz * kz;
    // r and p of a round's results are requested before its butterfly
    constexpr int RL = FxPlan<N>::r3 > 1 ? FxPlan<N>::r3 : FxPlan<N>::r2;
    double2 rpre[RL], ppre[RL];
    auto request = [&](int m) {
#pragma unroll
      for (int i = 0; i < RL; ++i) {
        const size_t e = base + (size_t)ln_index<N, FxPlan<N>>(t, m * RL + i) * rowstride;
        rpre[i] = r[e];
        ppre[i] = __ldg(p + e);
      }
    };
    ln_forward<N, FxPlan<N>, -1>(v, slots + l, ColMap<NL>{}, t, tw, [&](int k, fxc X, int i) {
      if (kz == 0) return;
      const int kxs = sfreq(k, N), n2 = kxs * kxs + k0;
      const size_t e = base + (size_t)k * rowstride;
      double2 rv = rpre[i % RL];
      const double2 pv = ppre[i % RL], tv = fx_to2(X, f);
      const double c = __ldg(ctab + n2);
      double2 q;
      if (UNIT_M) {
        q = make_double2(fma(c, tv.x, pv.x), fma(c, tv.y, pv.y));
      } else {
        const double m = __ldg(mtab + n2);
        q = make_double2(m * pv.x + c * tv.x, m * pv.y + c * tv.y);
      }
      rv.x -= alpha * q.x;
      rv.y -= alpha * q.y;
      r[e] = rv;
      const double m2 = rv.x * rv.x + rv.y * rv.y;
      rr += m2;
      rc = fma(cg_ic2<UNIT_M>(mtab, n2, c), m2, rc);
    }, request);
    rr *= 2.0;
    rc *= 2.0;
  } else {
    fxc* nat = reinterpret_cast<fxc*>(tw + N);  // both lines' T^ in natural order
    ln_forward<N, FxPlan<N>, -1>(v, slots + l, ColMap<NL>{}, t, tw, [&](int k, fxc X, int) {
      if (l < 2) nat[l * N + k] = X;
    });
    __syncthreads();
    if (l < 2 && !(l == 1 && row_y == ky))
      for (int k = t; k < N; k += N1) {
        const int kxs = sfreq(k, N), n2 = kxs * kxs + ky_s * ky_s;
        const size_t e = base + (size_t)k * rowstride;
        const double c0 = __ldg(ctab + n2), cN = __ldg(ctab + n2 + NH * NH);
        const double m0 = cg_m<UNIT_M>(mtab, n2), mN = cg_m<UNIT_M>(mtab, n2 + NH * NH);
        const double ca = 0.5 * (c0 + cN), cb = 0.5 * (c0 - cN), ma = 0.5 * (m0 + mN), mb = 0.5 * (m0 - mN);
        const double2 zc = fx_to2(nat[l * N + k], f), zp = fx_to2(nat[(1 - l) * N + (N - k) % N], f);
        const double2 pv = __ldg(p + e);
        double2 pp = make_double2(0.0, 0.0);
        if (mb != 0.0) pp = __ldg(p + (size_t)((N - row_y) % N) * NH + (size_t)((N - k) % N) * rowstride);
        double2 rv = r[e];
        rv.x -= alpha * (ma * pv.x + mb * pp.x + (ca * zc.x + cb * zp.x));
        rv.y -= alpha * (ma * pv.y - mb * pp.y + (ca * zc.y - cb * zp.y));
        r[e] = rv;
        const double m2 = rv.x * rv.x + rv.y * rv.y;
        rr += m2;
        rc = fma(fmax(cg_ic2<UNIT_M>(mtab, n2, c0), cg_ic2<UNIT_M>(mtab, n2 + NH * NH, cN)), m2, rc);
      }
  }
  const double s1 = block_sum(rr, red);
  const double s2 = block_sum(rc, red);
  if (tid == 0) {
    partials[0] = s1;
    partials[1] = s2;
  }
}

// z turn: each (x, y) line packed -> real, times D, -> packed; partial of D T^2.  grid (GZ, 1, systems)
template <int N>
__global__ void __launch_bounds__(FxZ<N>::NT)
k_fx_zturn(double2* __restrict__ spec, const double* __restrict__ D, const int4* __restrict__ twtab,
           double* __restrict__ partials, const CgScal* __restrict__ sc, Bat bt) {
  using G = FxZ<N>;
  constexpr int R1 = G::R1, N1 = G::N1, H = G::H;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  fxc* slots = reinterpret_cast<fxc*>(smem_raw);
  int4* tw = reinterpret_cast<int4*>(slots + G::NL * G::LS);
  __shared__ int se[2 * G::NL];
  __shared__ unsigned sq[2 * G::NL];
  __shared__ double red[32];
  const int z = blockIdx.z, tid = threadIdx.x, l = tid / N1, t = tid % N1;
  fx_load_tw<N>(tw, twtab, tid, G::NT);
  chain_start();
  if (sc && finished(sc + z)) return;
  const size_t row = (size_t)blockIdx.x * G::NL + l;
  double2* line = spec + z * bt.spec + row * H;
  double2 raw[R1];
#pragma unroll
  for (int r = 0; r < R1; ++r) raw[r] = line[r * N1 + t];
  for (int i = tid; i < 2 * G::NL; i += G::NT) {
    se[i] = FxScale::kMin;
    sq[i] = 0;
  }
  __syncthreads();
  const FxScale f = fx_line_scale<FxScale>(raw, &se[l], &sq[l], fx_c2r_count<N>());
  fxc* sl = slots + l * G::LS;
#pragma unroll
  for (int r = 0; r < R1; ++r) sl[PadMap{}(r * N1 + t)] = fx_from2(raw[r], f);
  __syncthreads();
  fxc v[R1];
  ln_inverse<H, FxPlan<H>, +1, 2>(v, sl, PadMap{}, t, tw, [&](int k) { return fx_c2r<N>(sl, PadMap{}, k, tw); });
  const double2* d = reinterpret_cast<const double2*>(D + z * bt.real) + row * H;
  double acc = 0.0;
#pragma unroll
  for (int r = 0; r < R1; ++r) {
    const double2 dv = __ldg(d + r * N1 + t), T = fx_to2(v[r], f);
    raw[r] = make_double2(T.x * dv.x, T.y * dv.y);
    acc = fma(raw[r].x, T.x, fma(raw[r].y, T.y, acc));
  }
  const FxScale g = fx_line_scale<FxScale>(raw, &se[G::NL + l], &sq[G::NL + l], H);
#pragma unroll
  for (int r = 0; r < R1; ++r) v[r] = fx_from2(raw[r], g);
  ln_forward_nat<H, FxPlan<H>, -1, 2>(v, sl, PadMap{}, t, tw);
  for (int k = t; k < H; k += N1) line[k] = fx_to2(fx_r2c<N>(sl, PadMap{}, k, tw), g);
  const double sum = block_sum(acc, red);
  if (tid == 0) partials[(size_t)z * bt.part + blockIdx.x] = sum;
}

}  // namespace wf
