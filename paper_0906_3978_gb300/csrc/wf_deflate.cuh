// wf_deflate.cuh -- two-level preconditioning of the inner CG by the lowest Fourier modes.
//
// The Wiener system is solved by CG in Fourier variables (Sec. 3.3.1); its slowest directions are
// the long-wavelength modes, where the prior S is largest and couples them through the survey
// mask.  The coarse space Z is spanned by the modes with |k|^2 <= K^2 (k in grid units), and
// E = Z^T A' Z is its Galerkin block of the preconditioned operator A' = C A C:
//     E(p, q) = m(p) delta_pq + c(p) c(q) Dh(p - q),   Dh = DFT of D = nbar w / V_c,
// a dense matrix built from the transform of the window at the differences of coarse modes.  Each
// inner CG runs preconditioned by the "A-DEF2" two-level operator of the deflation literature
// (Tang, Nabben, Vuik and Erlangga 2009, Sec. 2.3.3 there):
//     z = r - Z E^-1 Z^T (A' r - r),   started from x0 = Z E^-1 Z^T b (one step with alpha = 1),
// which, unlike plain deflated CG, keeps converging when E^-1 and A' r are only accurate to
// FP32.  E^-1 is formed once per solve by block Gauss-Jordan exchange in FP32.
//
// Coordinates.  A real field's spectrum is Hermitian, so the coarse space has nc = 2 nh + 1 real
// coordinates: k = 0 (the value y_0) and, for each of the nh half-space modes h (kz > 0, or
// kz = 0 with ky > 0, or kz = ky = 0 with kx > 0), a_h = sqrt2 Re y_h and b_h = sqrt2 Im y_h.  This
// basis is orthonormal for the CG inner product (the full-spectrum sum of Re(conj u v)).
//
// Per iteration (FP32 vectors, the packed half spectrum of wf_spectral.cuh):
//   k_xcr       T = IFFT_x(c r); then the solver's y pass, IFFT_y
//   k_zcoarse   IFFT_z, times D, FFT_z; keep kz <= K (the kz = 0 plane only)   -> Gz [N][N][K+1]
//   k_ycoarse   DFT along y at |ky| <= K                                      -> Gy [2K+1][K+1][N]
//   k_xcoarse   DFT along x at the coarse modes; g = coords of (m - 1) r + c Gc, and coords of r
//   k_defl_mu   mu = E^-1 g (one warp per mode); r -= Z mu kept aside for the x pass, which forms
//               p = (r - Z mu) + beta p; partials of <r, Z mu>
//               and, by its last CTA, <r, z> = <r, r> - <r, Z mu>; beta = <r, z> / <r, z>_prev; alpha's
//               numerator
//   (x pass 1)  then k_defl_alpha puts the saved coarse entries of r back
#pragma once
#include "wf_spectral.cuh"

namespace wf {

constexpr int kDeflTile = 64;   // block of the coarse Gauss-Jordan exchange

// packed-spectrum index of the signed mode (kx, ky, kz), 0 <= kz < N/2
template <int N> WF_D size_t dslot(int kx, int ky, int kz) {
  return ((size_t)((kx + N) % N) * N + (size_t)((ky + N) % N)) * (N / 2) + kz;
}

// ------------------------------------------------------------------------------------------
// x stage of the coarse projection: T = IFFT_x(c (.) r), the first pass of the inverse transform
// of c r (the CG x pass 1 without its vector updates: r and the table gathers in flight together,
// the packed column combined with its partner line at -ky).  grid (N/2 / NL, N, systems).
// ------------------------------------------------------------------------------------------
template <class R, int N, int RMAX = 8>
__global__ void __launch_bounds__(XYG<R, N>::NT)
k_xcr(const typename Store<R>::T* __restrict__ r, typename Store<R>::T* __restrict__ T,
      const typename Store<R>::S* __restrict__ ctab, const typename Store<R>::T* __restrict__ twtab,
      const CgScal* __restrict__ sc, Bat bt) {
  using G = XYG<R, N>;
  using SS = typename Store<R>::S;
  using VT = typename G::VT;
  constexpr int NH = G::NH;
  static_assert(std::is_same<R, SS>::value, "the CG passes compute in their storage type");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  cx<R>* tile = reinterpret_cast<cx<R>*>(smem_raw);
  cx<R>* tw = tile + G::M * G::LD;
  const int z = blockIdx.z;
  chain_start();
  if (finished(sc + z)) return;
  r += z * bt.spec;
  T += z * bt.spec;
  ctab += z * bt.tab;
  const int tid = threadIdx.x;
  const int kz0 = blockIdx.x * G::NL, ky = blockIdx.y;
  const int ky_s = sfreq(ky, N);
  load_tw<R, G::M, 2 * N>(tw, twtab, tid, G::NT);
  const size_t rowstride = (size_t)N * NH;
  const size_t base = (size_t)ky * NH + kz0;
  constexpr int CH = 4;
#pragma unroll
  for (int k0 = 0; k0 < G::PER; k0 += CH) {
    VT rv[CH];
    SS cv[CH][G::VW];
#pragma unroll
    for (int k = 0; k < CH && k0 + k < G::PER; ++k) {
      const int idx = tid + (k0 + k) * G::NT;
      if (G::EVEN || idx < G::NVEC) {
        const int i = idx / G::NV, c0 = (idx % G::NV) * G::VW;
        rv[k] = *reinterpret_cast<const VT*>(r + base + (size_t)i * rowstride + c0);
        const int kxs = sfreq(i, N);
#pragma unroll
        for (int u = 0; u < G::VW; ++u) {
          const int kz = kz0 + c0 + u;
          cv[k][u] = ctab[kxs * kxs + ky_s * ky_s + kz * kz];
        }
      }
    }
#pragma unroll
    for (int k = 0; k < CH && k0 + k < G::PER; ++k) {
      const int idx = tid + (k0 + k) * G::NT;
      if (G::EVEN || idx < G::NVEC) {
        const int i = idx / G::NV, c0 = (idx % G::NV) * G::VW;
        SS* rs = reinterpret_cast<SS*>(&rv[k]);
#pragma unroll
        for (int u = 0; u < G::VW; ++u)
          if (kz0 + c0 + u != 0) {  // column kz = 0 stays raw for the packed-column combine
            rs[2 * u] *= cv[k][u];
            rs[2 * u + 1] *= cv[k][u];
          }
        vec_to_tile<G>(tile, i, c0, rv[k]);
      }
    }
  }
  if (kz0 == 0) {  // partner line of column 0: r at (kx, -ky, 0)
    const size_t pb = (size_t)((N - ky) % N) * NH;
    for (int i = tid; i < G::M; i += G::NT) tile[i * G::LD + G::NL] = ld_c<R>(r + pb + (size_t)i * rowstride);
  }
  __syncthreads();
  if (kz0 == 0) combine_col0<R, N, G::LD, G::NL>(tile, ky_s, ctab, tid, G::NT);
  fft_line<R, G::M, G::TPL, G::LD, +1, 1, cmin(RMAX, rmax_for(G::M, G::TPL))>(tile + tid % G::NL, tid / G::NL, tw);
  tile_store<G>(tile, T + base, rowstride, tid);
}

// ------------------------------------------------------------------------------------------
// z stage of the coarse projection (the z turn without its full store): each (x, y) line of the
// y-transformed field is taken to real space, multiplied by D, transformed forward, and its
// kz = 0..K coefficients are stored; element 0 keeps only the kz = 0 plane (its real part), so the
// later x / y DFTs give that plane's coefficients directly.  grid (N*N / NL, 1, systems).
// ------------------------------------------------------------------------------------------
template <class R, int N>
__global__ void __launch_bounds__(ZG<R, N>::NT)
k_zcoarse(const typename Store<R>::T* __restrict__ spec, const typename Store<R>::S* __restrict__ D,
          const typename Store<R>::T* __restrict__ twtab, typename Store<R>::T* __restrict__ gz, int K,
          const CgScal* __restrict__ sc, Bat bt, size_t gzs) {
  using G = ZG<R, N>;
  using SS = typename Store<R>::S;
  static_assert(std::is_same<R, SS>::value, "the CG passes compute in their storage type");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  cx<R>* tile = reinterpret_cast<cx<R>*>(smem_raw);
  cx<R>* tw = tile + G::M * G::LD;  // 2N entries
  const int z = blockIdx.z;
  chain_start();
  if (finished(sc + z)) return;
  spec += z * bt.spec;
  D += z * bt.real;
  gz += z * gzs;
  const int tid = threadIdx.x;
  const size_t row0 = (size_t)blockIdx.x * G::NL;
  if (tid < G::NL) prefetch_l2(D + (row0 + tid) * N, N * sizeof(SS));
  for (int e = tid; e < 2 * N; e += G::NT) tw[e] = ld_c<R>(twtab + e);
  zrows_load<G>(tile, spec, row0, tid);
  __syncthreads();
  const int l = tid % G::NL, t = tid / G::NL;
  c2r_prep<R, N, G::LD>(tile + l, t, G::TPL, tw);
  __syncthreads();
  fft_line<R, G::M, G::TPL, G::LD, +1, 4, rmax_for(G::M, G::TPL)>(tile + l, t, tw);
  // real samples 2i, 2i+1 of line l sit in element i
#pragma unroll 4
  for (int k = 0; k < G::PER; ++k) {
    const int idx = tid + k * G::NT;
    if (!(G::EVEN || idx < G::NVEC)) continue;
    const int ll = idx / G::NV, i = (idx % G::NV) * G::VW;
    const SS* dp = D + (row0 + ll) * N + 2 * i;
    if constexpr (G::VW == 2) {
      const float4 d = *reinterpret_cast<const float4*>(dp);
      cx<R> a = tile[i * G::LD + ll], b = tile[(i + 1) * G::LD + ll];
      a.x = a.x * RT<R>::from_f(d.x);
      a.y = a.y * RT<R>::from_f(d.y);
      b.x = b.x * RT<R>::from_f(d.z);
      b.y = b.y * RT<R>::from_f(d.w);
      tile[i * G::LD + ll] = a;
      tile[(i + 1) * G::LD + ll] = b;
    } else {
      const double2 d = *reinterpret_cast<const double2*>(dp);
      cx<R> a = tile[i * G::LD + ll];
      a.x = a.x * RT<R>::c(d.x);
      a.y = a.y * RT<R>::c(d.y);
      tile[i * G::LD + ll] = a;
    }
  }
  __syncthreads();
  fft_line<R, G::M, G::TPL, G::LD, -1, 4, rmax_for(G::M, G::TPL)>(tile + l, t, tw);
  r2c_post<R, N, G::LD>(tile + l, t, G::TPL, tw);
  __syncthreads();
  for (int e = tid; e < G::NL * (K + 1); e += G::NT) {
    const int ll = e / (K + 1), i = e % (K + 1);
    cx<R> v = tile[i * G::LD + ll];
    if (i == 0) v.y = RT<R>::c(0.0);  // drop the kz = N/2 plane packed beside kz = 0
    st_c(gz + (row0 + ll) * (K + 1) + i, v);
  }
}

// ------------------------------------------------------------------------------------------
// y stage: Gy[ky + K][kz][x] = sum_y exp(-2 pi i ky y / N) Gz[x][y][kz] for |ky| <= K.
// With n3 > 0 one more CTA takes beta and the stop test of the iteration before from its n3 pairs of partial sums
// (nothing before this kernel uses them; a launch of its own costs 3 us, and in k_xcr the sums' code took the registers
// of its loads in flight: 512^3 solve 382 ms, here 344).
// grid (N + (n3 > 0), systems), 256 threads; shared memory N (K + 1) + N complex values.
// ------------------------------------------------------------------------------------------
template <class R, int N>
__global__ void __launch_bounds__(256)
k_ycoarse(const typename Store<R>::T* __restrict__ gz, const typename Store<R>::T* __restrict__ twtab,
          typename Store<R>::T* __restrict__ gy, int K, CgScal* __restrict__ sc, size_t gzs, size_t gys, Bat bt,
          const double* __restrict__ part, int n3, double inv_vc) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int KZ = K + 1;
  cx<R>* a = reinterpret_cast<cx<R>*>(smem_raw);  // [N][K+1]
  cx<R>* tw = a + N * KZ;                          // tw[e] = exp(-2 pi i e / N)
  const int z = blockIdx.y;
  for (int e = threadIdx.x; e < N; e += blockDim.x) tw[e] = ld_c<R>(twtab + 2 * e);
  chain_start();
  if (finished(sc + z)) return;
  int x = blockIdx.x;
  if (n3 > 0 && x-- == 0) {
    fin_beta(part + (size_t)z * bt.part, n3, inv_vc, sc + z, reinterpret_cast<double*>(smem_raw));
    return;
  }
  gz += z * gzs + (size_t)x * N * KZ;
  gy += z * gys;
  for (int e = threadIdx.x; e < N * KZ; e += blockDim.x) a[e] = ld_c<R>(gz + e);
  __syncthreads();
  const int nout = (2 * K + 1) * KZ;
  for (int o = threadIdx.x; o < nout; o += blockDim.x) {
    const int ky = o / KZ - K, kz = o % KZ;
    const int step = (ky + N) % N;
    R sr = RT<R>::c(0.0), si = RT<R>::c(0.0);
    int e = 0;
    for (int y = 0; y < N; ++y) {
      const cx<R> v = a[y * KZ + kz], w = tw[e];
      sr += v.x * w.x - v.y * w.y;
      si += v.x * w.y + v.y * w.x;
      e += step;
      if (e >= N) e -= N;
    }
    st_c(gy + (size_t)o * N + x, cx<R>{sr, si});
  }
}

// ------------------------------------------------------------------------------------------
// x stage and coordinates: one warp per half-space mode (warp nh: k = 0).
// MODE 0: gco = rco = coordinates of r (the start, x0 = Z E^-1 Z^T r).
// MODE 1: Gc = sum_x exp(-2 pi i kx x / N) Gy[ky + K][kz][x];  w = (m - 1) r + c Gc;
//         gco = coordinates of w (= Z^T (A' r - r)), rco = coordinates of r.
// r on the kz = 0 plane is unpacked from the column pair: r0(h) = (Z(h) + conj Z(-h)) / 2.
// grid (ceil((nh + 1) / 8), systems), 256 threads.
// ------------------------------------------------------------------------------------------
template <class R, int N, int MODE>
__global__ void __launch_bounds__(256)
k_xcoarse(const typename Store<R>::T* __restrict__ gy, const typename Store<R>::T* __restrict__ r,
          const typename Store<R>::S* __restrict__ ctab, const typename Store<R>::S* __restrict__ mtab,
          const typename Store<R>::T* __restrict__ twtab, const int4* __restrict__ modes, int nh, int K,
          float* __restrict__ gco, float* __restrict__ rco, const CgScal* __restrict__ sc, Bat bt, size_t gys,
          int ncp) {
  const int z = blockIdx.y;
  chain_start();
  if (finished(sc + z)) return;
  const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (warp > nh) return;
  r += z * bt.spec;
  ctab += z * bt.tab;
  mtab += z * bt.tab;
  gy += z * gys;
  gco += (size_t)z * ncp;
  rco += (size_t)z * ncp;
  int4 md = make_int4(0, 0, 0, 0);
  if (warp < nh) md = modes[warp];
  const cx<R> v1 = ld_c<R>(r + dslot<N>(md.x, md.y, md.z));
  cx<R> rh = v1;
  if (md.z == 0) {
    const cx<R> v2 = ld_c<R>(r + dslot<N>(-md.x, -md.y, 0));
    const R h = RT<R>::c(0.5);
    rh = cx<R>{(v1.x + v2.x) * h, (v1.y - v2.y) * h};
  }
  R gr = RT<R>::c(0.0), gi = RT<R>::c(0.0);
  if constexpr (MODE == 1) {
    const typename Store<R>::T* line = gy + (size_t)((md.y + K) * (K + 1) + md.z) * N;
    const int step = (md.x + N) % N;
    const int step32 = (int)(((long long)step * 32) % N);
    int e = (int)(((long long)step * lane) % N);
    for (int xx = lane; xx < N; xx += 32) {
      const cx<R> v = ld_c<R>(line + xx), w = ld_c<R>(twtab + 2 * e);
      gr += v.x * w.x - v.y * w.y;
      gi += v.x * w.y + v.y * w.x;
      e += step32;
      if (e >= N) e -= N;
    }
    for (int o = 16; o > 0; o >>= 1) {
      gr += __shfl_xor_sync(0xffffffffu, gr, o);
      gi += __shfl_xor_sync(0xffffffffu, gi, o);
    }
  }
  if (lane != 0) return;
  R wr = rh.x, wi = rh.y;
  if constexpr (MODE == 1) {
    const R c = tab_to<R>(ctab[md.w]), m1 = tab_to<R>(mtab[md.w]) - RT<R>::c(1.0);
    wr = m1 * rh.x + c * gr;
    wi = m1 * rh.y + c * gi;
  }
  const float s2 = 1.41421356237309505f;
  if (warp < nh) {
    gco[1 + 2 * warp] = s2 * (float)wr;
    gco[2 + 2 * warp] = s2 * (float)wi;
    rco[1 + 2 * warp] = s2 * (float)rh.x;
    rco[2 + 2 * warp] = s2 * (float)rh.y;
  } else {
    gco[0] = (float)wr;
    rco[0] = (float)rh.x;
  }
}

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

// alpha, and the coarse entries of r back to what k_defl_mu<MODE 1> saved (x pass 1 has used its own); grid = systems
template <class R, int N>
__global__ void k_defl_alpha(YFin fin, CgScal* sc, Bat bt) {
  __shared__ double red[32];
  const int z = blockIdx.x;
  chain_start();
  if (finished(sc + z)) return;
  for (int u = threadIdx.x; u <= fin.nh; u += blockDim.x)
    restore_entry<N>(fin.r + z * bt.spec, fin.rsave + (size_t)z * (2 * fin.nh + 1), fin.modes, fin.nh, u);
  fin_alpha(fin.part + (size_t)z * bt.part, fin.n1, fin.off, fin.n2, sc + z, red);
}

// <r, z> = <r, r> - <r, Z mu> (sc->rr holds <r, r> from the last x pass 2); beta = <r, z> over its
// previous value (0 on the first iteration after the start step); alpha's numerator becomes <r, z>.
WF_D void fin_defl(const double* dpart, int nh, CgScal* sc, double* red) {
  const double s = sum_fresh(dpart, nh + 1, 1, red);
  if (threadIdx.x == 0) {
    const double rz = sc->rr - s;
    if (!(rz > 0.0) || !isfinite(rz)) {
      sc->done = 3;
      return;
    }
    sc->beta = sc->defl == 1 ? 0.0 : rz / sc->rzo;
    if (sc->defl == 1) sc->defl = 0;
    sc->rzo = rz;
    sc->rr = rz;
  }
}

// ------------------------------------------------------------------------------------------
// mu = E^-1 g, one warp per half-space mode (rows 1 + 2j, 2 + 2j; warp nh: row 0), and its use
// (mu = 0 for a system with off[z] or its noco set):
// MODE 0: vec (zeroed) receives Z mu (the start vector).
// MODE 1: the coarse entries of vec (= r) are saved to rsave and replaced by r - Z mu; the
//         partial <r, Z mu> = rco . mu of the warp goes to dpart[warp].
// Z mu has (a + i b) / sqrt2 at h and its conjugate at -h (stored on the kz = 0 plane only).
// grid (ceil((nh + 1) / 8), systems), 256 threads, ncp floats of shared memory.
// ------------------------------------------------------------------------------------------
template <class R, int N, int MODE>
__global__ void __launch_bounds__(256)
k_defl_mu(const float* __restrict__ Einv, const float* __restrict__ gco, const float* __restrict__ rco,
          const int4* __restrict__ modes, int nh, int ncp, typename Store<R>::T* __restrict__ vec,
          typename Store<R>::T* __restrict__ rsave, double* __restrict__ dpart, CgScal* __restrict__ sc,
          Bat bt, const int* __restrict__ off) {
  __shared__ double red[32];
  using ST = typename Store<R>::T;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* gs = reinterpret_cast<float*>(smem_raw);
  const int z = blockIdx.y;
  chain_start();
  if (finished(sc + z)) return;
  Einv += (size_t)z * ncp * ncp;
  gco += (size_t)z * ncp;
  rco += (size_t)z * ncp;
  vec += z * bt.spec;
  rsave += (size_t)z * (2 * nh + 1);
  dpart += (size_t)z * (nh + 1);
  for (int e = threadIdx.x; e < ncp; e += blockDim.x) gs[e] = gco[e];
  __syncthreads();
  const int warp = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)), lane = threadIdx.x & 31;
  auto product = [&] {
    if (warp > nh) return;
    const int ra = warp < nh ? 1 + 2 * warp : 0;
    const float4* rowa = reinterpret_cast<const float4*>(Einv + (size_t)ra * ncp);
    const float4* rowb = reinterpret_cast<const float4*>(Einv + (size_t)(ra + 1) * ncp);
    const float4* g4 = reinterpret_cast<const float4*>(gs);
    // The products are summed exactly in double-float: the rows of E^-1 cancel heavily against g
    // (its weak directions carry entries up to 1/lambda_min), and an FP32 sum of nc terms loses
    // ~sqrt(nc) u of the terms' magnitude, which an ill-conditioned E turns into a stalled CG.
    // one accumulator per vector component (four independent chains per row); the loads of four
    // vectors of each row are issued before their products, to keep enough of them in flight
    AccF aa[4], ab[4];
    const bool two = warp < nh;
    constexpr int U = 4;
    const int nq = ncp / 4;  // a multiple of 32: ncp is a multiple of 128
    for (int q0 = lane; q0 < nq; q0 += 32 * U) {
      float4 av[U], bv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int q = q0 + 32 * u;
        av[u] = q < nq ? __ldg(rowa + q) : make_float4(0.f, 0.f, 0.f, 0.f);
        bv[u] = (two && q < nq) ? __ldg(rowb + q) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int q = q0 + 32 * u;
        if (q >= nq) break;
        const float4 g = g4[q];
        aa[0].add_prod(av[u].x, g.x);
        aa[1].add_prod(av[u].y, g.y);
        aa[2].add_prod(av[u].z, g.z);
        aa[3].add_prod(av[u].w, g.w);
        if (two) {
          ab[0].add_prod(bv[u].x, g.x);
          ab[1].add_prod(bv[u].y, g.y);
          ab[2].add_prod(bv[u].z, g.z);
          ab[3].add_prod(bv[u].w, g.w);
        }
      }
    }
    double da = (aa[0].get() + aa[1].get()) + (aa[2].get() + aa[3].get());
    double db = (ab[0].get() + ab[1].get()) + (ab[2].get() + ab[3].get());
    for (int o = 16; o > 0; o >>= 1) {
      da += __shfl_xor_sync(0xffffffffu, da, o);
      db += __shfl_xor_sync(0xffffffffu, db, o);
    }
    // a system whose coarse block failed the condition guard (k_defl_guard), or whose deflated inner
    // solve failed (noco, set by the host), gets mu = 0: plain CG
    const bool plain = off[z] || sc[z].noco;
    const float sa = plain ? 0.f : (float)da, sb = plain ? 0.f : (float)db;
    if (lane != 0) return;
    if (warp < nh) {
      const int4 md = modes[warp];
      const float h = 0.70710678118654752f;
      const cx<R> v{RT<R>::from_f(sa * h), RT<R>::from_f(sb * h)};
      const size_t s1 = dslot<N>(md.x, md.y, md.z);
      const size_t s2 = dslot<N>(-md.x, -md.y, 0);
      if constexpr (MODE == 0) {
        st_c(vec + s1, v);
        if (md.z == 0) st_c(vec + s2, conj(v));
      } else {
        dpart[warp] = (double)rco[ra] * (double)sa + (double)rco[ra + 1] * (double)sb;
        const ST o1 = vec[s1];
        rsave[2 * warp] = o1;
        st_c(vec + s1, ld_c<R>(&o1) - v);
        if (md.z == 0) {
          const ST o2 = vec[s2];
          rsave[2 * warp + 1] = o2;
          st_c(vec + s2, ld_c<R>(&o2) - conj(v));
        }
      }
    } else {
      const cx<R> v{RT<R>::from_f(sa), RT<R>::c(0.0)};
      if constexpr (MODE == 0) {
        st_c(vec, v);
      } else {
        dpart[nh] = (double)rco[0] * (double)sa;
        const ST o = vec[0];
        rsave[2 * nh] = o;
        st_c(vec, ld_c<R>(&o) - v);
      }
    }
  };
  product();
  if constexpr (MODE == 1) {  // the last CTA takes <r, z> and beta
    __syncthreads();          // every warp's entry of dpart
    if (last_cta(&sc[z].tick, gridDim.x)) fin_defl(dpart, nh, sc + z, red);
  }
}

// arm the start step (alpha = 1) of every running system; grid = systems
static __global__ void k_defl_arm(CgScal* sc) {
  sc += blockIdx.x;
  if (threadIdx.x == 0 && sc->done == 0) sc->defl = 2;
}

// ------------------------------------------------------------------------------------------
// Set-up: the transform of D at the differences of coarse modes, the coarse matrix, its inverse.
// ------------------------------------------------------------------------------------------
// DH[(dx + 2K) C^2 + (dy + 2K) C + dz + 2K] = scale * What(dx, dy, dz), C = 4K + 1, |d.| <= 2K,
// from the packed spectrum What of w (negative dz by conjugate symmetry, dz = 0 unpacked from the
// column pair); scale = nbar / V_c turns it into the transform of D.  grid (ceil(C^3 / 256), systems)
template <class R, int N>
__global__ void k_dh_gather(const typename Store<R>::T* __restrict__ what, float2* __restrict__ dh, int K,
                            double inv_vc, const CgScal* __restrict__ sc, Bat bt) {
  const int z = blockIdx.y;
  const int C = 4 * K + 1;
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= C * C * C) return;
  what += z * bt.spec;
  dh += (size_t)z * C * C * C;
  const int dx = i / (C * C) - 2 * K, dy = (i / C) % C - 2 * K, dz = i % C - 2 * K;
  cx<R> v;
  if (dz > 0) {
    v = ld_c<R>(what + dslot<N>(dx, dy, dz));
  } else if (dz < 0) {
    v = conj(ld_c<R>(what + dslot<N>(-dx, -dy, -dz)));
  } else {
    const cx<R> a = ld_c<R>(what + dslot<N>(dx, dy, 0)), b = ld_c<R>(what + dslot<N>(-dx, -dy, 0));
    const R h = RT<R>::c(0.5);
    v = cx<R>{(a.x + b.x) * h, (a.y - b.y) * h};
  }
  const double s = sc[z].nbar * inv_vc;
  dh[i] = make_float2((float)((double)v.x * s), (float)((double)v.y * s));
}

// E[i][j] over the coarse coordinates (identity on the padding [nc, ncp)):
//   (0, 0)      m0 + c0^2 Dh(0)
//   (0, a|b h)  sqrt2 c0 c_h Re|Im Dh(h)
//   (a h, a h') m_h [h = h'] + c c' (Re Dh(h - h') + Re Dh(h + h'))
//   (a h, b h') c c' (Im Dh(h + h') - Im Dh(h - h'))
//   (b h, a h') c c' (Im Dh(h - h') + Im Dh(h + h'))
//   (b h, b h') m_h [h = h'] + c c' (Re Dh(h - h') - Re Dh(h + h'))
// E is symmetric to the last bit: the tiles above the diagonal are computed (their FP64 products bound the kernel) and
// written twice.  grid (ncp / 16, ncp / 16, systems), 16 x 16 threads
template <class S>
__global__ void k_ebuild(const float2* __restrict__ dh, const S* __restrict__ ctab, const S* __restrict__ mtab,
                         const int4* __restrict__ modes, int nh, int ncp, int K, float* __restrict__ E, int tabs) {
  const int z = blockIdx.z;
  const int C = 4 * K + 1;
  if (blockIdx.y > blockIdx.x) return;
  __shared__ float tile[16][17];
  const int i = blockIdx.y * 16 + threadIdx.y, j = blockIdx.x * 16 + threadIdx.x;
  dh += (size_t)z * C * C * C;
  ctab += (size_t)z * tabs;
  mtab += (size_t)z * tabs;
  E += (size_t)z * ncp * ncp;
  const int nc = 2 * nh + 1;
  auto D = [&](int x, int y, int w) { return dh[((x + 2 * K) * C + (y + 2 * K)) * C + (w + 2 * K)]; };
  const double s2 = 1.41421356237309505;
  double v;
  if (i >= nc || j >= nc) {
    v = i == j ? 1.0 : 0.0;
  } else if (i == 0 && j == 0) {
    v = (double)mtab[0] + (double)ctab[0] * (double)ctab[0] * (double)D(0, 0, 0).x;
  } else if (i == 0 || j == 0) {
    const int c = i == 0 ? j : i;
    const int4 h = modes[(c - 1) / 2];
    const float2 d = D(h.x, h.y, h.z);
    v = s2 * (double)ctab[0] * (double)ctab[h.w] * (double)(((c - 1) % 2) == 0 ? d.x : d.y);
  } else {
    const int u = (i - 1) / 2, u2 = (j - 1) / 2, pi = (i - 1) % 2, pj = (j - 1) % 2;
    const int4 h = modes[u], g = modes[u2];
    const float2 A = D(h.x - g.x, h.y - g.y, h.z - g.z), B = D(h.x + g.x, h.y + g.y, h.z + g.z);
    const double cc = (double)ctab[h.w] * (double)ctab[g.w];
    const double dg = u == u2 ? (double)mtab[h.w] : 0.0;
    if (pi == 0 && pj == 0) v = dg + cc * ((double)A.x + (double)B.x);
    else if (pi == 0) v = cc * ((double)B.y - (double)A.y);
    else if (pj == 0) v = cc * ((double)A.y + (double)B.y);
    else v = dg + cc * ((double)A.x - (double)B.x);
  }
  E[(size_t)i * ncp + j] = (float)v;
  if (blockIdx.y == blockIdx.x) return;
  tile[threadIdx.y][threadIdx.x] = (float)v;
  __syncthreads();
  E[(size_t)(blockIdx.x * 16 + threadIdx.y) * ncp + blockIdx.y * 16 + threadIdx.x] = tile[threadIdx.x][threadIdx.y];
}

// Condition guard.  A coarse block built and inverted in FP32 cannot hold a condition number far
// beyond 1/u.  With the signal-dependent noise of sparse Jackknife subsamples (128^3, |k| <= 4 or 6),
// blocks with kappa_inf(E) of 8e8 and more stalled or broke down the deflated CG, while blocks up to
// 6e7 mostly converge 2-4x faster (below 1e8 kappa alone does not decide: a few failed from 1.4e7).
// Systems above kDeflCondMax run as plain CG (mu = 0); the plain filter's blocks sit near 1e3-1e4.
constexpr double kDeflCondMax = 1e8;
// Iteration cap of one deflated inner solve.  Deflated inner solves take ~40-50 iterations at 512^3
// and up to a few hundred on the Jackknife subsamples; one that reaches the cap (or breaks down)
// has lost the coarse space's benefit, and the system's later inner solves run as plain CG.
constexpr int kDeflInnerCap = 1200;
// max over the rows of one warp-group of the row sums of |M|; grid (ncp / 8, systems), 256 threads:
// one warp per row, the CTA's maximum to part[z * (ncp / 8) + blockIdx.x]
static __global__ void __launch_bounds__(256) k_defl_rownorm(const float* __restrict__ M, int ncp,
                                                             double* __restrict__ part) {
  __shared__ double red[8];
  const int z = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * 8 + warp;
  const float* m = M + (size_t)z * ncp * ncp + (size_t)row * ncp;
  double acc = 0.0;
  for (int j = lane; j < ncp; j += 32) acc += fabs((double)m[j]);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) red[warp] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double mx = red[0];
    for (int w = 1; w < 8; ++w) mx = fmax(mx, red[w]);
    part[(size_t)z * (ncp / 8) + blockIdx.x] = mx;
  }
}
// off[z] = 1 when kappa_inf = ||E||_inf ||E^-1||_inf exceeds kDeflCondMax or is not finite; grid =
// systems, 256 threads
static __global__ void k_defl_guard(const double* __restrict__ pe, const double* __restrict__ pi, int ncp,
                                    int* __restrict__ off) {
  __shared__ double r1[256], r2[256];
  const int z = blockIdx.x, nblk = ncp / 8;
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < nblk; i += blockDim.x) {
    a = fmax(a, pe[(size_t)z * nblk + i]);
    b = fmax(b, pi[(size_t)z * nblk + i]);
  }
  r1[threadIdx.x] = a;
  r2[threadIdx.x] = b;
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) {
      r1[threadIdx.x] = fmax(r1[threadIdx.x], r1[threadIdx.x + h]);
      r2[threadIdx.x] = fmax(r2[threadIdx.x], r2[threadIdx.x + h]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double k = r1[0] * r2[0];
    off[z] = (isfinite(k) && k <= kDeflCondMax) ? 0 : 1;
  }
}

// Block Gauss-Jordan exchange on block row / column kb of the SPD matrix M (ncp x ncp, row-major;
// after every block of the diagonal is exchanged, M holds M^-1):
//   P = M_kk^-1;  M_kj <- -P M_kj;  M_ik <- M_ik P;  M_ij <- M_ij - M_ik P M_kj  (i, j != k).
// No pivoting: every diagonal block of an SPD matrix's successive Schur complements is SPD.
// Step kb: k_gj_panel forms the block row and saves the old block column; k_gj_update updates every
// other block, and its first CTA, which takes the next diagonal block (kb + 1, kb + 1), also exchanges
// that block once updated (the next step's P), so that serial work overlaps the update.  P alternates
// between two buffers: step kb reads P[kb & 1] while the next one is written.

// exchange of the 64 x 64 block a (row stride LDA) in shared memory by the NT threads of the CTA; a
// becomes its inverse.  The same block Gauss-Jordan exchange one level down: for each of the four
// 16 x 16 diagonal sub-blocks, exchange it element by element (16 short serial steps), form its
// sub-row, save its old sub-column, and update the rest by rank-16 products, so the serial steps
// touch 256 elements instead of 4096.  cbuf holds 2 x 64 x 16 floats.  Every thread of the CTA calls it.
template <int NT, int LDA>
WF_D void gj_exchange64(float* a, float* cbuf) {
  constexpr int B = kDeflTile, S = 16;
  static_assert((S * S) % NT == 0 || NT > S * S, "threads");
  constexpr int PER = NT >= S * S ? 1 : S * S / NT;
  const int tid = threadIdx.x;
  for (int s0 = 0; s0 < B; s0 += S) {
    // (i) the diagonal sub-block, element by element
    for (int k = s0; k < s0 + S; ++k) {
      const float inv = 1.f / a[k * LDA + k];
      float nv[PER];
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        const int e = tid + q * NT, i = s0 + e / S, j = s0 + e % S;
        float v = 0.f;
        if (e < S * S) {
          if (i == k && j == k) v = inv;
          else if (i == k) v = -a[k * LDA + j] * inv;
          else if (j == k) v = a[i * LDA + k] * inv;
          else v = a[i * LDA + j] - a[i * LDA + k] * (a[k * LDA + j] * inv);
        }
        nv[q] = v;
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        const int e = tid + q * NT;
        if (e < S * S) a[(s0 + e / S) * LDA + s0 + e % S] = nv[q];
      }
      __syncthreads();
    }
    // (ii) old sub-column C(i, :) = a[i][s0..s0+S) for i outside the sub-block, kept in cbuf
    for (int e = tid; e < B * S; e += NT) {
      const int i = e / S, c = e % S;
      cbuf[e] = (i >= s0 && i < s0 + S) ? 0.f : a[i * LDA + s0 + c];
    }
    __syncthreads();
    // (iii) sub-row R = P a[sub][j] (P = the exchanged sub-block), written as -R; j outside
    for (int e = tid; e < S * B; e += NT) {
      const int r = e / B, j = e % B;
      if (j >= s0 && j < s0 + S) continue;
      float acc = 0.f;
#pragma unroll
      for (int c = 0; c < S; ++c) acc = fmaf(a[(s0 + r) * LDA + s0 + c], a[(s0 + c) * LDA + j], acc);
      cbuf[B * S + e] = acc;  // R(r, j)
    }
    __syncthreads();
    for (int e = tid; e < S * B; e += NT) {
      const int r = e / B, j = e % B;
      if (j >= s0 && j < s0 + S) continue;
      a[(s0 + r) * LDA + j] = -cbuf[B * S + e];
    }
    // (iv) every element outside the sub-block's rows: a[i][j] -= C(i, :) R(:, j) for j outside its
    // columns, a[i][j] = C(i, :) P(:, j) inside them
    for (int e = tid; e < B * B; e += NT) {
      const int i = e / B, j = e % B;
      if (i >= s0 && i < s0 + S) continue;
      float acc = 0.f;
      if (j >= s0 && j < s0 + S) {
#pragma unroll
        for (int c = 0; c < S; ++c) acc = fmaf(cbuf[i * S + c], a[(s0 + c) * LDA + j], acc);
        a[i * LDA + j] = acc;
      } else {
#pragma unroll
        for (int c = 0; c < S; ++c) acc = fmaf(cbuf[i * S + c], cbuf[B * S + c * B + j], acc);
        a[i * LDA + j] -= acc;
      }
    }
    __syncthreads();
  }
}

// (0) the first diagonal block; grid (1, 1, systems), 64 threads
static __global__ void __launch_bounds__(64) k_gj_pivot(float* __restrict__ M, float* __restrict__ P, int ncp) {
  constexpr int B = kDeflTile;
  __shared__ __align__(16) float a[B][68];
  __shared__ float cbuf[2 * B * 16];
  const int z = blockIdx.z;
  M += (size_t)z * ncp * ncp;
  P += (size_t)z * 2 * B * B;  // buffer 0 of the system's pair
  for (int e = threadIdx.x; e < B * B; e += blockDim.x) a[e / B][e % B] = M[(size_t)(e / B) * ncp + e % B];
  __syncthreads();
  gj_exchange64<64, 68>(&a[0][0], cbuf);
  for (int e = threadIdx.x; e < B * B; e += blockDim.x) {
    M[(size_t)(e / B) * ncp + e % B] = a[e / B][e % B];
    P[e] = a[e / B][e % B];
  }
}

// 64 x 64 x 64 product on 64 threads (8 x 8 outputs each): acc += As^T Bs with As[k][i] = A(i, k)
// and Bs[k][j] = B(k, j), rows of 68 floats.
WF_D void gj_tile_mma(const float (*As)[68], const float (*Bs)[68], float acc[8][8], int ty, int tx) {
#pragma unroll 4
  for (int k = 0; k < kDeflTile; ++k) {
    const float4 a0 = *reinterpret_cast<const float4*>(&As[k][ty * 8]);
    const float4 a1 = *reinterpret_cast<const float4*>(&As[k][ty * 8 + 4]);
    const float4 b0 = *reinterpret_cast<const float4*>(&Bs[k][tx * 8]);
    const float4 b1 = *reinterpret_cast<const float4*>(&Bs[k][tx * 8 + 4]);
    const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
  }
}

WF_D void l2_hint(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// load a 64 x 64 block (row stride ld) into shared memory, transposed (T = true: S[c][r] = G(r, c))
// or not, as float4 rows
template <bool T>
WF_D void gj_load(float (*S)[68], const float* __restrict__ G, size_t ld) {
  for (int e = threadIdx.x; e < kDeflTile * kDeflTile / 4; e += blockDim.x) {
    const int r = e / (kDeflTile / 4), c = (e % (kDeflTile / 4)) * 4;
    const float4 v = *reinterpret_cast<const float4*>(G + (size_t)r * ld + c);
    if (T) {
      S[c][r] = v.x;
      S[c + 1][r] = v.y;
      S[c + 2][r] = v.z;
      S[c + 3][r] = v.w;
    } else {
      *reinterpret_cast<float4*>(&S[r][c]) = v;
    }
  }
}

// (1) the block row: Rp_j = P M_kj (kept for (2)), M_kj <- -Rp_j; and the old block column
// Cp_j = M_jk copied aside.  grid (ncp / 64, 1, systems), 64 threads.
static __global__ void __launch_bounds__(64) k_gj_panel(float* __restrict__ M, const float* __restrict__ P,
                                                        float* __restrict__ Rp, float* __restrict__ Cp, int ncp,
                                                        int kb) {
  constexpr int B = kDeflTile;
  __shared__ __align__(16) float As[B][68];
  __shared__ __align__(16) float Bs[B][68];
  const int z = blockIdx.z, jb = blockIdx.x;
  if (jb == kb) return;
  M += (size_t)z * ncp * ncp;
  P += (size_t)z * 2 * B * B + (size_t)(kb & 1) * B * B;
  Rp += (size_t)z * B * ncp;
  Cp += (size_t)z * ncp * B;
  float* Mkj = M + (size_t)kb * B * ncp + (size_t)jb * B;
  const float* Mjk = M + (size_t)jb * B * ncp + (size_t)kb * B;
  gj_load<true>(As, P, B);      // As[k][i] = P(i, k)
  gj_load<false>(Bs, Mkj, ncp);  // Bs[k][j] = M_kj(k, j)
  for (int e = threadIdx.x; e < B * B / 4; e += blockDim.x) {
    const int r = e / (B / 4), c = (e % (B / 4)) * 4;
    *reinterpret_cast<float4*>(Cp + ((size_t)jb * B + r) * B + c) =
        *reinterpret_cast<const float4*>(Mjk + (size_t)r * ncp + c);
  }
  __syncthreads();
  const int ty = threadIdx.x / 8, tx = threadIdx.x % 8;
  float acc[8][8] = {};
  gj_tile_mma(As, Bs, acc, ty, tx);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = ty * 8 + i;
    float* rp = Rp + (size_t)r * ncp + (size_t)jb * B + tx * 8;
    float* mk = Mkj + (size_t)r * ncp + tx * 8;
    *reinterpret_cast<float4*>(rp) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    *reinterpret_cast<float4*>(rp + 4) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
    *reinterpret_cast<float4*>(mk) = make_float4(-acc[i][0], -acc[i][1], -acc[i][2], -acc[i][3]);
    *reinterpret_cast<float4*>(mk + 4) = make_float4(-acc[i][4], -acc[i][5], -acc[i][6], -acc[i][7]);
  }
}

// (2) every block (ib, jb), ib != kb: M_ib,jb -= Cp_ib Rp_jb, or M_ib,kb = Cp_ib P, as 128 x 128
// tiles of 2 x 2 blocks (256 threads, 8 x 8 outputs each).  The first CTA takes the tile that holds
// the next diagonal block (kb + 1, kb + 1) (the tile it would have had goes to that tile's CTA) and,
// once its update is done, exchanges that block in shared memory, writing the next P.
// grid (ncp / 128, ncp / 128, systems), 256 threads, UPD_SMEM bytes of dynamic shared memory.
constexpr int kUpdLd = 2 * kDeflTile + 4;  // 132: float4 rows, banks spread
constexpr size_t kUpdSmem = (size_t)2 * kDeflTile * kUpdLd * sizeof(float);
static __global__ void __launch_bounds__(256) k_gj_update(float* __restrict__ M, float* __restrict__ P,
                                                          const float* __restrict__ Rp, const float* __restrict__ Cp,
                                                          int ncp, int kb) {
  constexpr int B = kDeflTile, T2 = 2 * B, LD = kUpdLd;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* As = reinterpret_cast<float*>(smem_raw);  // [64 k][132]: As[k][i] = A(i, k), i < 128
  float* Bs = As + B * LD;                          // [64 k][132]: Bs[k][j] = B(k, j), j < 128
  const int z = blockIdx.z, ntl = ncp / T2, d = kb + 1;
  int tj = blockIdx.x, ti = blockIdx.y;
  const bool has_next = d < ncp / B;
  if (has_next) {  // swap the first CTA with the one of the tile holding block (d, d)
    if (ti == 0 && tj == 0) ti = tj = d / 2;
    else if (ti == d / 2 && tj == d / 2) ti = tj = 0;
  }
  (void)ntl;
  M += (size_t)z * ncp * ncp;
  float* Pn = P + (size_t)z * 2 * B * B + (size_t)(d & 1) * B * B;
  P += (size_t)z * 2 * B * B + (size_t)(kb & 1) * B * B;
  Rp += (size_t)z * B * ncp;
  Cp += (size_t)z * ncp * B;
  const int tid = threadIdx.x;
  // the tile itself, read at the end: asked into L2 now (M is larger than L2)
  for (int e = tid; e < T2 * T2 / 32; e += 256)
    l2_hint(M + ((size_t)ti * T2 + e / (T2 / 32)) * ncp + (size_t)tj * T2 + (e % (T2 / 32)) * 32);
  // A: the old block columns of the tile's two block rows (Cp rows), transposed into As
  for (int e = tid; e < T2 * B / 4; e += 256) {
    const int r = e / (B / 4), c = (e % (B / 4)) * 4;  // r < 128: row of the tile, c: k
    const float4 v = *reinterpret_cast<const float4*>(Cp + ((size_t)ti * T2 + r) * B + c);
    As[(c + 0) * LD + r] = v.x;
    As[(c + 1) * LD + r] = v.y;
    As[(c + 2) * LD + r] = v.z;
    As[(c + 3) * LD + r] = v.w;
  }
  // B: for each of the tile's two block columns, the block row Rp_jb, or P where jb = kb
  for (int e = tid; e < B * T2 / 4; e += 256) {
    const int k = e / (T2 / 4), c = (e % (T2 / 4)) * 4;  // c < 128: column of the tile
    const int jb = tj * 2 + c / B, cc = c % B;
    const float4 v = jb == kb ? *reinterpret_cast<const float4*>(P + (size_t)k * B + cc)
                              : *reinterpret_cast<const float4*>(Rp + (size_t)k * ncp + (size_t)jb * B + cc);
    *reinterpret_cast<float4*>(&Bs[k * LD + c]) = v;
  }
  __syncthreads();
  const int ty = tid / 16, tx = tid % 16;
  float acc[8][8] = {};
#pragma unroll 4
  for (int k = 0; k < B; ++k) {
    const float4 a0 = *reinterpret_cast<const float4*>(&As[k * LD + ty * 8]);
    const float4 a1 = *reinterpret_cast<const float4*>(&As[k * LD + ty * 8 + 4]);
    const float4 b0 = *reinterpret_cast<const float4*>(&Bs[k * LD + tx * 8]);
    const float4 b1 = *reinterpret_cast<const float4*>(&Bs[k * LD + tx * 8 + 4]);
    const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
  }
  // the thread's 8 x 8 outputs lie in one block (ib, jb)
  const int ib = ti * 2 + (ty * 8) / B, jb = tj * 2 + (tx * 8) / B;
  const bool diag_tile = has_next && ti == d / 2 && tj == d / 2;
  const bool diag = diag_tile && ib == d && jb == d;
  if (diag_tile) __syncthreads();  // As / Bs are reused for the block below
  if (ib != kb) {
    float* Tb = M + (size_t)(ti * T2 + ty * 8) * ncp + (size_t)tj * T2 + tx * 8;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float* t = Tb + (size_t)i * ncp;
      float4 v0 = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      float4 v1 = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
      if (jb != kb) {
        const float4 o0 = *reinterpret_cast<const float4*>(t), o1 = *reinterpret_cast<const float4*>(t + 4);
        v0 = make_float4(o0.x - v0.x, o0.y - v0.y, o0.z - v0.z, o0.w - v0.w);
        v1 = make_float4(o1.x - v1.x, o1.y - v1.y, o1.z - v1.z, o1.w - v1.w);
      }
      if (diag) {  // the block (d, d) goes to shared memory, rows of 68
        const int r = (ty * 8) % B + i, c = (tx * 8) % B;
        *reinterpret_cast<float4*>(&As[r * 68 + c]) = v0;
        *reinterpret_cast<float4*>(&As[r * 68 + c + 4]) = v1;
      } else {
        *reinterpret_cast<float4*>(t) = v0;
        *reinterpret_cast<float4*>(t + 4) = v1;
      }
    }
  }
  if (!diag_tile) return;
  __syncthreads();
  gj_exchange64<256, 68>(As, Bs);
  float* Td = M + (size_t)d * B * ncp + (size_t)d * B;
  for (int e = tid; e < B * B; e += 256) {
    const float v = As[(e / B) * 68 + e % B];
    Td[(size_t)(e / B) * ncp + e % B] = v;
    Pn[e] = v;
  }
}

}  // namespace wf
