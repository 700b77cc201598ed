// wf_solver_impl.cuh -- drivers of the Wiener solve (Kitaura et al. 2009, Sec. 3.3.1, Eq. eq:WF).
//
// System: A s = b with A = S^-1 + diag(nbar w), S^-1 = F^-1 diag(dV/P(k)) F, b = R^T N^-1 d.
//
// The iteration runs in Fourier variables.  With C = F^-1 diag(c) F a real, even Fourier
// multiplier, CG is applied to (C A C) y = C b and s = C y; the CG vectors are stored as
// packed half spectra (the DFT of the real-space vectors).  In those variables
//     (C A C) y^ = m (.) y^ + c (.) F( D (.) F^-1 (c (.) y^) ),   D = nbar w,
// with m = c^2 S^-1.  precond = 1 takes c = S^(1/2) (m = 1 except at k = 0, where
// c_0 = (nbar sum(w)/V_c)^(-1/2) and m_0 = 0); precond = 0 takes c = 1, m = S^-1, which is
// textbook CG on A itself.  Either way the stop test is on the canonical residual b - A s:
// its norm is estimated every iteration from the preconditioned residual (||C^-1 r~||) and,
// once the estimate is below tol, recomputed in FP64 from s.
//
// One CG iteration = 5 FFT passes (17 spectra of traffic):
//   x pass 1: p = r + beta p, x += alpha_prev p_old, T = IFFT_x(c p)
//   y pass  : IFFT_y
//   z turn  : IFFT_z, times D / V_c, FFT_z
//   y pass  : FFT_y
//   finisher: alpha = rr / <p, A p> (<p, m p> from x pass 1, <c p, D c p> from the z turn)
//   x pass 2: FFT_x, q = m p + c T, r -= alpha q, <r, r>, ||C^-1 r||^2 (q is never stored)
// (for FP32 at the sizes plane_cs() lists, the three middle passes run as one thread-block
// cluster kernel per x-plane, k_plane_turn)
//   finisher: beta, stop test
#pragma once
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <cmath>
#include <vector>

#include "wf_ctx.h"
#include "wf_solver_group.h"
#include "wf_plane.cuh"
#include "wf_spectral.cuh"
#include "wf_fixspec.cuh"
#include "wf_deflate.cuh"

namespace wf {

// Arithmetic of the FP64-storage passes.  Their transforms run in 64-bit fixed point (wf_fix.cuh), the
// vector updates and sums in FP64.
using FP64Arith = double;

template <class K>
static inline cudaError_t set_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Launch geometry and launchers of the spectral passes for one arithmetic type and size; every
// launcher covers `nb` systems laid out with the strides `bt` (blockIdx.z = system).
template <class R, int N>
struct Spec {
  using ST = typename Store<R>::T;
  using SS = typename Store<R>::S;
  static constexpr int NH = N / 2;
  static constexpr int NLxy = XYG<R, N>::NL;
  static_assert(NH % NLxy == 0 && (N * N) % tile_lines<R>() == 0, "tile widths must divide the grid");
  static constexpr int NTy = XYG<R, N>::NT;
  static constexpr int NTx = XYG<R, N>::NT;
  static constexpr size_t SMxy = XYG<R, N>::SMEM;
  static constexpr int NLz = ZG<R, N>::NL;
  static constexpr int NTz = ZG<R, N>::NT;
  static constexpr size_t SMz = ZG<R, N>::SMEM;
  static constexpr int GXY = (NH / NLxy) * N;   // blocks of an x or y pass (per system)
  static constexpr int GZ = N * N / NLz;        // blocks of a z pass (per system)
  static constexpr bool F64 = sizeof(SS) == 8;  // FP64 storage: fixed-point transforms
  using FC = FxC<N>;
  using FZ = FxZ<N>;
  static constexpr int GXF = F64 ? (FC::KB + 1) * N : GXY;  // partial sums of the CG start's x pass
  static constexpr int GZI = F64 ? FZ::GZ : GZ;             // partial sums of the z turn and the z inverse
  // The FP64 residual of a mixed solve runs in FP64 butterflies up to 72^3 (all of it is 0.1 ms of a 4 ms solve at
  // 64^3).  Small boxes are where weak directions are common, and there the last inner solve may resolve one of
  // them or stop before it does, by the last bits of the residual it starts from: 1 of 219 drawn maps ended 4 times
  // as far from the converged one (8e-6) with the fixed-point residual, none above 72^3.
  static constexpr bool BUTTERFLY_RESID = F64 && N <= 72;
  static constexpr size_t SPEC = (size_t)N * N * NH;  // complex elements of a spectrum
  static constexpr size_t V = (size_t)N * N * N;
  static constexpr int TAB = 3 * (N / 2) * (N / 2) + 1;
  // partial sums per system.  An x pass writes one (the first) or two (the second) per tile, at
  // most NX tiles whatever its variant; the middle passes (z turn or plane kernel) write theirs
  // from offset NX.
  static constexpr int NX = N * NH;
  static constexpr int NMID = GZ > N * 8 ? GZ : N * 8;
  static constexpr int NPART = NX + NMID > 2 * NX ? NX + NMID : 2 * NX;
  static dim3 gxy(int nb) { return dim3(NH / NLxy, N, nb); }
  static dim3 gz(int nb) { return dim3(GZ, 1, nb); }
  static Bat bat() { return Bat{SPEC, V, TAB, NPART}; }

  // launch-profile class of a pass: FP64-storage launches (the solves' FP64 residuals, the FP64
  // solve) are kept apart from the FP32 inner passes of the same name
  static const char* cls(const char* f32, const char* f64) { return sizeof(SS) == 8 ? f64 : f32; }
  // algorithmic bytes of one launch per system (DRAM traffic the pass cannot avoid)
  static constexpr double BS = (double)SPEC * sizeof(ST);
  static constexpr double BV = (double)V;
  // cluster size of the fused y / z / y plane kernel (0: not available at this size)
  static constexpr int PCS = plane_cs<R, N>(), PE = plane_e<R, N>();
  // the persistent passes with tensor copies: tile lines and buffers in flight
  static constexpr int NLT = tma_lines<R, N>();

  static cudaError_t attrs() {
    static bool done = false;
    if (done) return cudaSuccess;
    cudaError_t e = cudaSuccess;
#define WF_A(k, b) if (e == cudaSuccess) e = set_smem(k, b)
    if constexpr (F64) {
      WF_A((k_fx_xmul<N>), fx_xmul_smem<N>());
      WF_A((k_fx_xfwd<N>), fx_xmul_smem<N>());
      WF_A((k_fx_xinv<N>), FC::SMEM);
      WF_A((k_fx_zfwd<N>), FZ::SMEM);
      WF_A((k_fx_zinv<N, ZI_STORE>), FZ::SMEM);
      WF_A((k_fx_zinv<N, ZI_RESID>), FZ::SMEM);
      if (e == cudaSuccess) e = YFix<FxWide>::setup();
      if constexpr (BUTTERFLY_RESID) {
        WF_A((k_zfwd<R, N>), SMz);
        WF_A((k_xmul<R, N, true, true, false>), SMxy);
        WF_A((k_zinv<R, N, ZI_RESID>), SMz);
        if (e == cudaSuccess) e = YV<NLT, 2, 8>::setup();
      }
    } else {
      WF_A((k_xmul<R, N, true, false, true>), SMxy);
      WF_A((k_xmul<R, N, false, true, false>), SMxy);
      WF_A((k_zfwd<R, N>), SMz);
      WF_A((k_zinv<R, N, ZI_ACCUM>), SMz);
    }
    if constexpr (std::is_same<R, float>::value) {
      WF_A((k_zcoarse<R, N>), SMz);
      WF_A((k_xcr<R, N, 32>), SMxy);
      WF_A(k_gj_update, kUpdSmem);
      WF_A((k_ycoarse<R, N>), (size_t)N * (kDeflMaxRadius + 2) * sizeof(cx<R>));
    }
    if constexpr (PCS > 0) WF_A((k_plane_turn<R, N, PCS, PE>), (PlaneG<R, N, PCS, PE>::SMEM));
#undef WF_A
    for (const PassVariant& v : yvariants())
      if (e == cudaSuccess) e = v.setup();
    for (const XVariant& v : xvariants())
      if (e == cudaSuccess) e = v.setup();
    for (const ZVariant& v : zvariants())
      if (e == cudaSuccess) e = v.setup();
    if (e == cudaSuccess) done = true;
    return e;
  }

  // persistent grid: every SM holds its resident CTAs, capped by the number of tiles
  static unsigned persistent_grid(const Ctx& c, int occ, long long tiles) {
    const long long g = (long long)occ * (c.sm_count > 0 ? c.sm_count : 152);
    return (unsigned)(tiles < g ? tiles : g);
  }
  // ---- launch variants of a pass (tile lines, buffers in flight, radix cap); the context's
  // tuning table picks one per (pass, precision, size), variant 0 by default ------------------
  using PassRun = void (*)(Ctx&, int, ST*, const ST*, CgScal*, int, cudaStream_t, const YFin&);
  struct PassVariant {
    const char* name;
    cudaError_t (*setup)();
    PassRun go;
    void run(Ctx& c, int nb, ST* t, const ST* tw, CgScal* sc, int dir, cudaStream_t st) const {
      go(c, nb, t, tw, sc, dir, st, YFin{});
    }
  };
  // alpha (and the coarse entries of r back) in launches of their own, for a middle pass that does not take them along
  static void finish_alpha(Ctx& c, int nb, CgScal* sc, const YFin& fin, cudaStream_t st) {
    if (fin.n1 <= 0) return;
    c.launch("fin", 0, st, [&] {
      if constexpr (!F64)
        if (fin.nh >= 0) return Ctx::chain(k_defl_alpha<float, N>, nb, 1024, 0, st, fin, sc, bat());
      Ctx::chain(k_fin_alpha, nb, 1024, 0, st, fin.part, fin.n1, fin.off, fin.n2, sc, bat());
    });
  }
  static void finish_beta(Ctx& c, int nb, double* part, int n3, double inv_vc, CgScal* sc, cudaStream_t st) {
    c.launch("fin", 0, st, [&] { Ctx::chain(k_fin_beta, nb, 1024, 0, st, part, n3, inv_vc, sc, bat()); });
  }
  // y pass variant <NL, STG, RMAX>: complex FFT along y of every (x, kz) line, in place
  template <int NL, int STG, int RMAX>
  struct YV {
    using G = TG<R, N, NL, STG>;
    static inline int occ = 1;  // resident CTAs per SM
    static cudaError_t setup() {
      cudaError_t e = set_smem(k_ypass_tma<R, N, -1, NL, STG, RMAX>, G::SMEM);
      if (e == cudaSuccess) e = set_smem(k_ypass_tma<R, N, +1, NL, STG, RMAX>, G::SMEM);
      if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_ypass_tma<R, N, -1, NL, STG, RMAX>, G::NT, G::SMEM);
      if (occ < 1) occ = 1;
      return e;
    }
    static void run(Ctx& c, int nb, ST* t, const ST* tw, CgScal* sc, int dir, cudaStream_t st, const YFin& fin) {
      CUtensorMap m;
      if (!make_spectrum_map(&m, t, N, nb, sizeof(SS) == 8, NL, G::BR, 1)) {
        c.map_failed = true;
        return;
      }
      const unsigned grid = persistent_grid(c, occ, (long long)nb * G::TPS);
      finish_alpha(c, nb, sc, fin, st);
      c.launch(cls("ypass", "ypass_f64"), 2 * BS * nb, st, [&] {
        if (dir < 0) Ctx::chain(k_ypass_tma<R, N, -1, NL, STG, RMAX>, grid, G::NT, G::SMEM, st, m, tw, sc, nb, c.dev_err);
        else Ctx::chain(k_ypass_tma<R, N, +1, NL, STG, RMAX>, grid, G::NT, G::SMEM, st, m, tw, sc, nb, c.dev_err);
      });
    }
  };
  // the FP64 y pass (fixed point); tw is unused, its twiddles come from the context
  template <class S>
  struct YFix {
    static cudaError_t setup() {
      cudaError_t e = set_smem(k_fx_ypass<N, -1, S>, FC::SMEM);
      return e == cudaSuccess ? set_smem(k_fx_ypass<N, +1, S>, FC::SMEM) : e;
    }
    static void run(Ctx& c, int nb, ST* t, const ST*, CgScal* sc, int dir, cudaStream_t st, const YFin& fin) {
      double2* T = reinterpret_cast<double2*>(t);
      const dim3 grid(FC::KB, N + (fin.n1 > 0), nb);
      c.launch("ypass_f64", 2 * BS * nb, st, [&] {
        if (dir < 0) Ctx::chain(k_fx_ypass<N, -1, S>, grid, FC::NT, FC::SMEM, st, T, c.fixed(N), sc, bat(), fin);
        else Ctx::chain(k_fx_ypass<N, +1, S>, grid, FC::NT, FC::SMEM, st, T, c.fixed(N), sc, bat(), fin);
      });
    }
  };
  static const std::vector<PassVariant>& yvariants() {
    static const std::vector<PassVariant> v = [] {
      std::vector<PassVariant> out;
      if constexpr (F64) {
        out.push_back({"fixed", YFix<FxScale>::setup, YFix<FxScale>::run});
      } else {
        // variant 0 decides how a mixed solve rounds (kInnerMargin): its radices stay
        out.push_back({"nl_s2_r8", YV<NLT, 2, 8>::setup, YV<NLT, 2, 8>::run});
        if constexpr (N >= 128) {
          constexpr int H = NLT / 2;
          out.push_back({"nl_s2_r32", YV<NLT, 2, 32>::setup, YV<NLT, 2, 32>::run});
          out.push_back({"nl_s3_r32", YV<NLT, 3, 32>::setup, YV<NLT, 3, 32>::run});
          out.push_back({"nl/2_s2_r32", YV<H, 2, 32>::setup, YV<H, 2, 32>::run});
          out.push_back({"nl/2_s3_r16", YV<H, 3, 16>::setup, YV<H, 3, 16>::run});
        }
      }
      return out;
    }();
    return v;
  }
  // ---- x-pass variants: the two CG x passes.  each launcher returns the number of partial sums it wrote
  using XinvRun = int (*)(Ctx&, int, ST*, ST*, ST*, ST*, ST*, const SS*, const SS*, bool, const ST*,
                          double*, CgScal*, cudaStream_t);
  using XupdRun = int (*)(Ctx&, int, const ST*, ST*, ST*, ST*, const SS*, const SS*, bool, const ST*,
                          double*, CgScal*, cudaStream_t);
  struct XVariant {
    const char* name;
    cudaError_t (*setup)();
    XinvRun xinv;
    XupdRun xupd;
  };
  // the register-staged kernels (one CTA per tile, loads through registers), radix cap RMAX
  template <int RMAX>
  struct XReg {
    static cudaError_t setup() {
      cudaError_t e = set_smem(k_cg_xinv<R, N, true, RMAX>, SMxy);
      if (e == cudaSuccess) e = set_smem(k_cg_xinv<R, N, false, RMAX>, SMxy);
      if (e == cudaSuccess) e = set_smem(k_cg_xupd<R, N, true, RMAX>, SMxy);
      if (e == cudaSuccess) e = set_smem(k_cg_xupd<R, N, false, RMAX>, SMxy);
      return e;
    }
    static int xinv(Ctx& c, int nb, ST* r, ST* P0, ST* P1, ST* x, ST* T, const SS* ctab, const SS* mtab, bool unit_m,
                    const ST* tw, double* part, CgScal* sc, cudaStream_t st) {
      c.launch("cg_xinv", 6 * BS * nb, st, [&] {
        if (unit_m)
          Ctx::chain(k_cg_xinv<R, N, true, RMAX>, gxy(nb), NTx, SMxy, st, r, P0, P1, x, T, ctab, mtab, tw, part, sc, bat());
        else
          Ctx::chain(k_cg_xinv<R, N, false, RMAX>, gxy(nb), NTx, SMxy, st, r, P0, P1, x, T, ctab, mtab, tw, part, sc, bat());
      });
      return GXY;
    }
    static int xupd(Ctx& c, int nb, const ST* T, ST* r, ST* P0, ST* P1, const SS* ctab, const SS* mtab, bool unit_m,
                    const ST* tw, double* part, CgScal* sc, cudaStream_t st) {
      c.launch("cg_xupd", 4 * BS * nb, st, [&] {
        if (unit_m)
          Ctx::chain(k_cg_xupd<R, N, true, RMAX>, gxy(nb), NTx, SMxy, st, T, r, P0, P1, ctab, mtab, tw, part, sc, bat());
        else
          Ctx::chain(k_cg_xupd<R, N, false, RMAX>, gxy(nb), NTx, SMxy, st, T, r, P0, P1, ctab, mtab, tw, part, sc, bat());
      });
      return GXY;
    }
  };
  // the FP64 CG x passes (fixed point)
  struct XFix {
    static cudaError_t setup() {
      cudaError_t e = set_smem(k_fx_cg_xinv<N, true>, FC::SMEM);
      if (e == cudaSuccess) e = set_smem(k_fx_cg_xinv<N, false>, FC::SMEM);
      if (e == cudaSuccess) e = set_smem(k_fx_cg_xupd<N, true>, fx_xmul_smem<N>());
      if (e == cudaSuccess) e = set_smem(k_fx_cg_xupd<N, false>, fx_xmul_smem<N>());
      return e;
    }
    static int xinv(Ctx& c, int nb, ST* r, ST* P0, ST* P1, ST* x, ST* T, const SS* ctab, const SS* mtab, bool unit_m,
                    const ST*, double* part, CgScal* sc, cudaStream_t st) {
      if constexpr (F64) {
        const dim3 grid(FC::KB, N, nb);
        c.launch("cg_xinv_f64", 6 * BS * nb, st, [&] {
          if (unit_m)
            Ctx::chain(k_fx_cg_xinv<N, true>, grid, FC::NT, FC::SMEM, st, r, P0, P1, x, T, ctab, mtab, c.fixed(N), part, sc, bat());
          else
            Ctx::chain(k_fx_cg_xinv<N, false>, grid, FC::NT, FC::SMEM, st, r, P0, P1, x, T, ctab, mtab, c.fixed(N), part, sc, bat());
        });
      }
      return FC::KB * N;
    }
    static int xupd(Ctx& c, int nb, const ST* T, ST* r, ST* P0, ST* P1, const SS* ctab, const SS* mtab, bool unit_m,
                    const ST*, double* part, CgScal* sc, cudaStream_t st) {
      if constexpr (F64) {
        const dim3 grid(FC::KB + 1, N, nb);
        const size_t sm = fx_xmul_smem<N>();
        c.launch("cg_xupd_f64", 4 * BS * nb, st, [&] {
          if (unit_m)
            Ctx::chain(k_fx_cg_xupd<N, true>, grid, FC::NT, sm, st, T, r, P0, P1, ctab, mtab, c.fixed(N), part, sc, bat());
          else
            Ctx::chain(k_fx_cg_xupd<N, false>, grid, FC::NT, sm, st, T, r, P0, P1, ctab, mtab, c.fixed(N), part, sc, bat());
        });
      }
      return (FC::KB + 1) * N;
    }
  };
  static const std::vector<XVariant>& xvariants() {
    static const std::vector<XVariant> v = [] {
      std::vector<XVariant> out;
      if constexpr (F64) {
        out.push_back({"fixed", XFix::setup, XFix::xinv, XFix::xupd});
      } else {
        out.push_back({"registers", XReg<8>::setup, XReg<8>::xinv, XReg<8>::xupd});
        if constexpr (N >= 128) {
          out.push_back({"registers_r16", XReg<16>::setup, XReg<16>::xinv, XReg<16>::xupd});
          out.push_back({"registers_r32", XReg<32>::setup, XReg<32>::xinv, XReg<32>::xupd});
        }
      }
      return out;
    }();
    return v;
  }
  // ---- z-turn variants: elements per thread (threads per CTA) ------------------------------
  using ZRun = int (*)(Ctx&, int, ST*, const SS*, const ST*, double*, const CgScal*, cudaStream_t);  // partial sums written
  struct ZVariant {
    const char* name;
    cudaError_t (*setup)();
    ZRun run;
  };
  template <int EZ>
  struct ZV {
    static cudaError_t setup() { return set_smem(k_zturn<R, N, EZ>, ZG<R, N, EZ>::SMEM); }
    static int run(Ctx& c, int nb, ST* T, const SS* D, const ST* tw, double* part, const CgScal* sc, cudaStream_t st) {
      using G = ZG<R, N, EZ>;
      c.launch("zturn", (2 * BS + sizeof(SS) * BV) * nb, st,
               [&] { Ctx::chain(k_zturn<R, N, EZ>, gz(nb), G::NT, G::SMEM, st, T, D, tw, part, sc, bat()); });
      return GZ;
    }
  };
  struct ZFix {  // FP64 (fixed point)
    static cudaError_t setup() { return set_smem(k_fx_zturn<N>, FZ::SMEM); }
    static int run(Ctx& c, int nb, ST* T, const SS* D, const ST*, double* part, const CgScal* sc, cudaStream_t st) {
      if constexpr (F64)
        c.launch("zturn_f64", (2 * BS + sizeof(SS) * BV) * nb, st,
                 [&] { Ctx::chain(k_fx_zturn<N>, dim3(FZ::GZ, 1, nb), FZ::NT, FZ::SMEM, st, T, D, c.fixed(N), part, sc, bat()); });
      return FZ::GZ;
    }
  };
  static const std::vector<ZVariant>& zvariants() {
    static const std::vector<ZVariant> v = [] {
      std::vector<ZVariant> out;
      if constexpr (F64) {
        out.push_back({"fixed", ZFix::setup, ZFix::run});
      } else {
        constexpr int E0 = z_elems<R, N>();
        out.push_back({"e_default", ZV<E0>::setup, ZV<E0>::run});
        if constexpr (N >= 128) {
          if constexpr (E0 / 2 >= 4 && (N / 2) % (E0 / 2) == 0) out.push_back({"e/2", ZV<E0 / 2>::setup, ZV<E0 / 2>::run});
          if constexpr (E0 / 4 >= 4 && (N / 2) % (E0 / 4) == 0) out.push_back({"e/4", ZV<E0 / 4>::setup, ZV<E0 / 4>::run});
        }
      }
      return out;
    }();
    return v;
  }
  static std::string tune_key(const char* pass) {
    return std::string(pass) + (sizeof(SS) == 8 ? "/f64/" : "/f32/") + std::to_string(N);
  }
  template <class V>
  static const V& pick(const Ctx& c, const char* pass, const std::vector<V>& vs) {
    auto it = c.tuned.find(tune_key(pass));
    const int i = it == c.tuned.end() ? 0 : it->second;
    return vs[i >= 0 && i < (int)vs.size() ? i : 0];
  }
  // complex FFT along y of every (x, kz) line of nb spectra, in place
  static void ypass(Ctx& c, int nb, ST* t, const ST* tw, CgScal* sc, int dir, cudaStream_t st, const YFin& fin = YFin{}) {
    pick(c, "ypass", yvariants()).go(c, nb, t, tw, sc, dir, st, fin);
  }
  // out = [IFFT_x] tab (.) [FFT_x] in (FP64 form with both transforms: fmul below)
  template <bool FWD, bool INV, bool DOT>
  static void xmul(Ctx& c, int nb, const ST* in, ST* out, const SS* tab, const ST* tw, double* part,
                   const CgScal* sc, cudaStream_t st) {
    c.launch(cls("xmul", "xmul_f64"), 2 * BS * nb, st, [&] {
      if constexpr (F64 && FWD) {
        static_assert(!INV && DOT, "the FP64 forward x pass starts a CG");
        k_fx_xfwd<N><<<dim3(FC::KB + 1, N, nb), FC::NT, fx_xmul_smem<N>(), st>>>(in, out, tab, c.fixed(N), part, bat());
      } else if constexpr (F64) {
        k_fx_xinv<N><<<dim3(FC::KB, N, nb), FC::NT, FC::SMEM, st>>>(in, out, tab, c.fixed(N), bat());
      } else {
        k_xmul<R, N, FWD, INV, DOT><<<gxy(nb), NTx, SMxy, st>>>(in, out, tab, tw, part, sc, bat());
      }
    });
  }
  // out = IFFT_x tab (.) FFT_x in in FP64 storage, tab as digits (k_table_digits), system z's power of two at
  // exps[z * estride]
  static void fmul(Ctx& c, int nb, const double2* in, double2* out, const double* tab, const int* exps, int estride,
                   cudaStream_t st) {
    c.launch("xmul_f64", 2 * BS * nb, st, [&] {
      k_fx_xmul<N><<<dim3(FC::KB + 1, N, nb), FC::NT, fx_xmul_smem<N>(), st>>>(
          in, out, reinterpret_cast<const int2*>(tab), exps, estride, c.fixed(N), bat());
    });
  }
  static void zfwd(Ctx& c, int nb, const double* in, ST* out, const ST* tw, const CgScal* sc, cudaStream_t st) {
    c.launch(cls("zfwd", "zfwd_f64"), (BS + 8 * BV) * nb, st, [&] {
      if constexpr (F64)
        k_fx_zfwd<N><<<dim3(FZ::GZ, 1, nb), FZ::NT, FZ::SMEM, st>>>(in, out, c.fixed(N), sc, bat());
      else k_zfwd<R, N><<<gz(nb), NTz, SMz, st>>>(in, out, tw, sc, bat());
    });
  }
  template <int MODE>
  static void zinv(Ctx& c, int nb, const ST* in, double* out, const double* s, const double* w, const double* b,
                   double scl, const ST* tw, double* part, const CgScal* sc, cudaStream_t st) {
    const double vb = MODE == ZI_RESID ? 4 : (MODE == ZI_ACCUM ? 2 : 1);
    c.launch(cls("zinv", "zinv_f64"), (BS + 8 * vb * BV) * nb, st, [&] {
      if constexpr (F64)
        k_fx_zinv<N, MODE><<<dim3(FZ::GZ, 1, nb), FZ::NT, FZ::SMEM, st>>>(in, out, s, w, b, scl, c.fixed(N), part, sc,
                                                                          bat());
      else k_zinv<R, N, MODE><<<gz(nb), NTz, SMz, st>>>(in, out, s, w, b, scl, tw, part, sc, bat());
    });
  }

  // res = b - (S^-1 + nbar diag(w)) s of a mixed solve (T, T2: scratch spectra; stab: the prior's table, FP64 values
  // with BUTTERFLY_RESID, else digits) and the partial sums of its squares, whose number is returned
  static int resid(Ctx& c, int nb, const double* s, const double* w, const double* b, double* res, ST* T, ST* T2,
                   const double* stab, const int* exps, int estride, double inv_vc, const ST* tw, double* part,
                   CgScal* sc, cudaStream_t st) {
    if constexpr (BUTTERFLY_RESID) {
      using Y = YV<NLT, 2, 8>;
      const Bat bt = bat();
      c.launch("zfwd_f64", (BS + 8 * BV) * nb, st,
               [&] { k_zfwd<R, N><<<gz(nb), NTz, SMz, st>>>(s, T, tw, nullptr, bt); });
      Y::run(c, nb, T, tw, nullptr, -1, st, YFin{});
      c.launch("xmul_f64", 2 * BS * nb, st, [&] {
        k_xmul<R, N, true, true, false><<<gxy(nb), NTx, SMxy, st>>>(T, T2, stab, tw, part, nullptr, bt);
      });
      Y::run(c, nb, T2, tw, nullptr, +1, st, YFin{});
      c.launch("zinv_f64", (BS + 8 * 4 * BV) * nb, st, [&] {
        k_zinv<R, N, ZI_RESID><<<gz(nb), NTz, SMz, st>>>(T2, res, s, w, b, inv_vc, tw, part, sc, bt);
      });
      return GZ;
    } else {
      zfwd(c, nb, s, T, tw, nullptr, st);
      ypass(c, nb, T, tw, nullptr, -1, st);
      fmul(c, nb, T, T2, stab, exps, estride, st);
      ypass(c, nb, T2, tw, nullptr, +1, st);
      zinv<ZI_RESID>(c, nb, T2, res, s, w, b, inv_vc, tw, part, sc, st);
      return GZI;
    }
  }

  // One CG iteration of every unfinished system (no host synchronisation).  The first x pass forms
  // p from rin (default r); fin: the coarse entries of r to put back (nh < 0: none), the rest is filled in here.
  // The number of partial sums of <r, r> and the estimate is returned; with `beta` they are taken here.
  static int iteration(Ctx& c, int nb, ST* r, ST* P0, ST* P1, ST* x, ST* T, const SS* D,
                       const SS* ctab, const SS* mtab, bool unit_m, const ST* tw, double* part, CgScal* sc, double inv_vc,
                       cudaStream_t st, ST* rin = nullptr, YFin fin = YFin{}, bool beta = true) {
    fin.part = part;
    fin.off = NX;
    fin.n1 = pick(c, "xinv", xvariants())
                 .xinv(c, nb, rin ? rin : r, P0, P1, x, T, ctab, mtab, unit_m, tw, part, sc, st);
    bool fused = false;
    if constexpr (PCS > 0) {
      if (c.fused_planes) {
        c.launch("plane_turn", (2 * BS + sizeof(SS) * BV) * nb, st,
                 [&] { plane_turn_launch<R, N, PCS, PE>(T, D, tw, part + NX, sc, bat(), nb, st); });
        fin.n2 = N * PCS;
        finish_alpha(c, nb, sc, fin, st);
        fused = true;
      }
    }
    if (!fused) {
      ypass(c, nb, T, tw, sc, +1, st);
      fin.n2 = pick(c, "zturn", zvariants()).run(c, nb, T, D, tw, part + NX, sc, st);
      ypass(c, nb, T, tw, sc, -1, st, fin);
    }
    const int n3 = pick(c, "xupd", xvariants()).xupd(c, nb, T, r, P0, P1, ctab, mtab, unit_m, tw, part, sc, st);
    if (beta) finish_beta(c, nb, part, n3, inv_vc, sc, st);
    return n3;
  }
};

// ---- small batched elementwise helpers (blockIdx.y = system) -----------------------------
// D = w * nbar / V_c (nbar from the system's scalars), in the type of the spectral arithmetic
template <class SSo>
__global__ void k_make_D(const double* __restrict__ w, SSo* __restrict__ D, const CgScal* __restrict__ sc,
                         double inv_vc, size_t n) {
  const int z = blockIdx.y;
  const double f = sc[z].nbar * inv_vc;
  w += z * n;
  D += z * n;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    D[i] = (SSo)(w[i] * f);
}
// partials[z * pstride + block] of sum(in) (SQ = false) or sum(in^2) (SQ = true).  Eight loads in flight per thread
// and six CTAs per SM: latency bound one of each (512^3: 1.60 ms, now under 0.32).
template <bool SQ>
__global__ void k_sum(const double* __restrict__ in, size_t n, double* __restrict__ partials, int pstride) {
  __shared__ double red[32];
  const int z = blockIdx.y;
  in += z * n;
  AccD acc;
  const size_t step = (size_t)gridDim.x * blockDim.x;
  size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  auto add = [&](double v) {
    if (SQ) acc.add_prod(v, v);
    else acc.add(v);
  };
  for (; i + 7 * step < n; i += 8 * step) {
    double v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = in[i + j * step];
#pragma unroll
    for (int j = 0; j < 8; ++j) add(v[j]);
  }
  for (; i < n; i += step) add(in[i]);
  const double s = block_sum(acc.get(), red);
  if (threadIdx.x == 0) partials[z * pstride + blockIdx.x] = s;
}

// Tables: ctab[n2] = c(k), mtab[n2] = c^2 S^-1 (k) for one system.
static void make_tables(const std::vector<double>& sinv, bool precond, double c0, double* ct, double* mt) {
  const size_t L = sinv.size();
  for (size_t i = 0; i < L; ++i) {
    if (!precond) {
      ct[i] = 1.0;
      mt[i] = sinv[i];
    } else if (i == 0) {
      ct[i] = c0;
      mt[i] = 0.0;
    } else {
      ct[i] = 1.0 / std::sqrt(sinv[i]);
      mt[i] = 1.0;
    }
  }
}

// Smallest e with every entry of v below 2^e in modulus (the power of two of a table's digits)
static inline int table_exp(const double* v, size_t n) {
  double m = 0.0;
  for (size_t i = 0; i < n; ++i) {
    if (!std::isfinite(v[i])) return kFxNanTab;
    m = std::max(m, std::fabs(v[i]));
  }
  int e = 0;
  std::frexp(m, &e);
  return e;
}

// Device table `name` from v, converted to T, through a page-locked staging buffer of the same
// name (an asynchronous copy: the staging buffer is rewritten only by a later solve of the same
// workspace, after this one's stream has finished).
template <class T>
static inline wf_status upload_tables(Ctx& c, const std::string& name, const std::vector<double>& v, T** out,
                                      cudaStream_t st) {
  T *h, *d;
  WF_TRY(c.get_pinned(name + "_stage", v.size() * sizeof(T), (void**)&h));
  for (size_t i = 0; i < v.size(); ++i) h[i] = (T)v[i];
  WF_TRY(c.get(name, v.size() * sizeof(T), (void**)&d));
  WF_CUDA(cudaMemcpyAsync(d, h, v.size() * sizeof(T), cudaMemcpyHostToDevice, st));
  *out = d;
  return WF_OK;
}

// ==========================================================================================
// A group: `nb` systems of one grid size and precision, solved together.  The host drives it
// as a state machine: enqueue() launches the next block of device work (ending with a copy of
// the scalars to pinned host memory), advance() consumes those scalars after the stream is
// synchronised and picks the next phase.
// ==========================================================================================

// Shared pieces: contiguous copies of w and b, sum(w), ||b||^2, tables, scalars.
template <int N>
struct GroupCommon : Group {
  static constexpr size_t V = (size_t)N * N * N;
  static constexpr int TAB = 3 * (N / 2) * (N / 2) + 1;
  std::string key;
  double *W = nullptr, *B = nullptr, *S = nullptr, *RES = nullptr, *part = nullptr;
  CgScal *sc = nullptr, *hsc = nullptr;
  const double2* tw = nullptr;
  std::vector<CgScal> h;       // host copy of the scalars
  std::vector<double> bb0, sumw, rel;
  std::vector<int> state;      // 0 running, 1 finished
  std::vector<int> bad;        // 1: rejected input (status already set)
  int phase = 0;
  double inv_vc = 1.0 / (double)V;
  // CUDA graph of one block of CG iterations (kernel arguments are fixed for the group)
  cudaGraphExec_t gexec = nullptr;
  long long glaunches = 0;

  ~GroupCommon() override {
    if (gexec) cudaGraphExecDestroy(gexec);
  }
  // Enqueue `body(stream)` on st: directly while the profiler times launches, otherwise as a
  // graph captured on the first call (on the context's capture stream) and replayed.
  template <class F>
  wf_status run_block(Ctx& c, cudaStream_t st, F&& body) {
    if (c.prof.on) {
      body(st);
      return WF_OK;
    }
    if (!gexec) {
      cudaStream_t cs;
      WF_TRY(c.capture_stream(&cs));
      const long long before = c.prof.launches;
      WF_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
      body(cs);
      cudaGraph_t g = nullptr;
      cudaError_t e = cudaStreamEndCapture(cs, &g);
      if (e == cudaSuccess) e = cudaGraphInstantiate(&gexec, g, 0);
      if (g) cudaGraphDestroy(g);
      glaunches = c.prof.launches - before;
      c.prof.launches = before;
      if (e != cudaSuccess) {
        gexec = nullptr;
        set_last_error("graph capture of the CG block", e);
        return WF_ERR_CUDA;
      }
    }
    WF_CUDA(cudaGraphLaunch(gexec, st));
    c.prof.launches += glaunches;
    return WF_OK;
  }

  // The prior's FP64 table `stab` (TAB entries per system) to digits in place, after push_scalars: the
  // systems' powers of two are in their scalars.
  void table_digits(Ctx& c, double* stab, cudaStream_t st) {
    c.launch("tables", 0, st, [&] {
      k_table_digits<<<dim3((TAB + 255) / 256, nb), 256, 0, st>>>(stab, TAB, &sc->texp, kScalInts);
    });
  }
  static constexpr int kScalInts = (int)(sizeof(CgScal) / sizeof(int));
  wf_status push_scalars(cudaStream_t st) {
    for (int m = 0; m < nb; ++m) hsc[m] = h[m];
    WF_CUDA(cudaMemcpyAsync(sc, hsc, nb * sizeof(CgScal), cudaMemcpyHostToDevice, st));
    return WF_OK;
  }
  wf_status pull_scalars(cudaStream_t st) {
    WF_CUDA(cudaMemcpyAsync(hsc, sc, nb * sizeof(CgScal), cudaMemcpyDeviceToHost, st));
    return WF_OK;
  }
  void read_scalars() { h.assign(hsc, hsc + nb); }
  bool all_done() const {
    for (int m = 0; m < nb; ++m)
      if (h[m].done == 0) return false;
    return true;
  }
};

// Per-system sums of w and b^2: two reductions, enqueued with the copy of the scalars back to the host (no synchronisation) ...
template <int N>
static wf_status group_sums_begin(Ctx& c, GroupCommon<N>& g, int npart, cudaStream_t st) {
  const size_t V = GroupCommon<N>::V;
  g.h.assign(g.nb, CgScal{});
  WF_TRY(g.push_scalars(st));
  const Bat b{0, 0, 0, npart};
  const int nblk = std::min(152 * 6, npart);  // partial sums fit a system's slots
  c.launch("reduce", 8.0 * V * g.nb, st, [&] { k_sum<false><<<dim3(nblk, g.nb), 256, 0, st>>>(g.W, V, g.part, npart); });
  c.launch("fin", 0, st, [&] { k_fin_sum<<<g.nb, 1024, 0, st>>>(g.part, nblk, 0, g.sc, b); });
  c.launch("reduce", 8.0 * V * g.nb, st, [&] { k_sum<true><<<dim3(nblk, g.nb), 256, 0, st>>>(g.B, V, g.part, npart); });
  c.launch("fin", 0, st, [&] { k_fin_sum<<<g.nb, 1024, 0, st>>>(g.part, nblk, 1, g.sc, b); });
  WF_CUDA(cudaGetLastError());
  return g.pull_scalars(st);
}
// ... and read once the stream has passed them.
template <int N>
static void group_sums_end(GroupCommon<N>& g) {
  g.read_scalars();
  g.sumw.resize(g.nb);
  g.bb0.resize(g.nb);
  g.bad.assign(g.nb, 0);
  for (int m = 0; m < g.nb; ++m) {
    g.sumw[m] = g.h[m].aux[0];
    g.bb0[m] = g.h[m].aux[1];
    // an empty window or a non-finite w or b is this system's argument error, not the batch's
    if (!(g.sumw[m] > 0.0) || !std::isfinite(g.sumw[m]) || !std::isfinite(g.bb0[m])) {
      g.bad[m] = 1;
      g.sumw[m] = 1.0;
      g.bb0[m] = 0.0;
      if (g.info[m]) *g.info[m] = wf_solve_info{0, 0, 0.0, g.sys[m]->nbar, WF_ERR_ARG};
    }
  }
}

// The last inner solve of a mixed solve aims at kInnerMargin x the remaining reduction (its stop
// test is an upper estimate of the canonical residual; the FP64 residual that follows decides).
// 0.9 saved ~2% of the iterations at 512^3 but moved the result from 5e-7 to 8e-7 of the solution
// converged to 1e-10, too close to the mixed path's 1e-6 bound.  The rule bounds the residual, not the error: in
// a system with weak directions (sparse surveys, boxes under ~200 Mpc/h; eigenvalues of 1e-3 and below beside 1) the
// map keeps what the rounding of the first inner solve left there, up to 2e-4 of it, and FP32 passes that
// round in another order (other radices, other groups of FP32 sums) or another margin leave something else.
constexpr double kInnerMargin = 0.5;

// Check interval: grids of 256^3 and up check the device flags every 4 iterations, smaller ones every 8 (a block
// of finished iterations still launches; a check costs ~15 us).
template <int N> constexpr int check_every() { return N >= 256 ? 4 : 8; }

// ------------------------------------------------------------------------------------------
// FP64 group: FP64 storage, spectral arithmetic R.
// Phases: 1 CG loop, 2 post (s = C x, explicit residual), 3 restart, 9 done.
// ------------------------------------------------------------------------------------------
template <class R, int N>
struct GroupFP64 : GroupCommon<N> {
  using SP = Spec<R, N>;
  using ST = typename Store<R>::T;
  using Base = GroupCommon<N>;
  using Base::nb; using Base::sys; using Base::info; using Base::key; using Base::W; using Base::B;
  using Base::S; using Base::RES; using Base::part; using Base::sc; using Base::tw; using Base::h;
  using Base::phase; using Base::inv_vc; using Base::bb0; using Base::rel; using Base::state;
  ST *xh, *rh, *P0, *P1, *T, *T2;
  double *D, *ct, *mt, *stab;
  std::vector<int> restarts;
  bool unit_m = true;

  wf_status prepare_begin(Ctx& c, cudaStream_t st) override {
    nb = (int)sys.size();
    key = this->tag + "f64_" + std::to_string(N) + "_";
    int* err;
    WF_TRY(c.err_word(&err));
    WF_CUDA(SP::attrs());
    const size_t SPEC = SP::SPEC, V = SP::V;
    WF_TRY(c.tw(N, &tw));
    WF_TRY(c.fix_tables(N));
    const char* nm[6] = {"x", "r", "p0", "p1", "T", "T2"};
    ST** ptr[6] = {&xh, &rh, &P0, &P1, &T, &T2};
    for (int i = 0; i < 6; ++i) WF_TRY(c.get(key + nm[i], nb * SPEC * sizeof(ST), (void**)ptr[i]));
    WF_TRY(c.get(key + "D", nb * V * sizeof(double), (void**)&D));
    WF_TRY(c.get(key + "W", nb * V * sizeof(double), (void**)&W));
    WF_TRY(c.get(key + "B", nb * V * sizeof(double), (void**)&B));
    WF_TRY(c.get(key + "S", nb * V * sizeof(double), (void**)&S));
    WF_TRY(c.get(key + "RES", nb * V * sizeof(double), (void**)&RES));
    WF_TRY(c.get(key + "part", (size_t)nb * SP::NPART * sizeof(double), (void**)&part));
    WF_TRY(c.get(key + "sc", nb * sizeof(CgScal), (void**)&sc));
    WF_TRY(c.get_pinned(key + "hsc", nb * sizeof(CgScal), (void**)&this->hsc));
    for (int m = 0; m < nb; ++m) {
      WF_CUDA(cudaMemcpyAsync(W + m * V, sys[m]->w, V * sizeof(double), cudaMemcpyDefault, st));
      WF_CUDA(cudaMemcpyAsync(B + m * V, sys[m]->b, V * sizeof(double), cudaMemcpyDefault, st));
    }
    return group_sums_begin<N>(c, *this, SP::NPART, st);
  }
  wf_status prepare_end(Ctx& c, cudaStream_t st) override {
    const size_t SPEC = SP::SPEC, V = SP::V;
    group_sums_end<N>(*this);
    // tables
    const int TAB = SP::TAB;
    std::vector<double> vc((size_t)nb * TAB), vm((size_t)nb * TAB), vs((size_t)nb * TAB);
    unit_m = true;
    for (int m = 0; m < nb; ++m) {
      const bool pre = sys[m]->opts.precond != 0;
      unit_m = unit_m && pre;
      const double c0 = 1.0 / std::sqrt(sys[m]->nbar * this->sumw[m] * inv_vc);
      make_tables(sys[m]->sinv, pre, c0, vc.data() + (size_t)m * TAB, vm.data() + (size_t)m * TAB);
      std::copy(sys[m]->sinv.begin(), sys[m]->sinv.end(), vs.begin() + (size_t)m * TAB);
    }
    if (unit_m)  // the FP64 CG passes take 1 / c^2 from the m table, whose values they know
      for (size_t i = 0; i < vm.size(); ++i) vm[i] = 1.0 / (vc[i] * vc[i]);
    WF_TRY(upload_tables<double>(c, key + "tc", vc, &ct, st));
    WF_TRY(upload_tables<double>(c, key + "tm", vm, &mt, st));
    WF_TRY(upload_tables<double>(c, key + "ts", vs, &stab, st));
    // scalars
    h.assign(nb, CgScal{});
    for (int m = 0; m < nb; ++m) {
      h[m].nbar = sys[m]->nbar;
      h[m].texp = table_exp(sys[m]->sinv.data(), TAB);
      h[m].max_iter = sys[m]->opts.max_iter;
      h[m].tol2 = sys[m]->opts.tol * sys[m]->opts.tol;
      h[m].bb = bb0[m];
      if (this->bad[m]) h[m].done = 4;
    }
    WF_TRY(this->push_scalars(st));
    this->table_digits(c, stab, st);
    c.launch("make_D", 16.0 * V * nb, st, [&] { k_make_D<double><<<dim3(152 * 4, nb), 256, 0, st>>>(W, D, sc, inv_vc, V); });
    WF_CUDA(cudaMemsetAsync(xh, 0, nb * SPEC * sizeof(ST), st));
    rel.assign(nb, 1.0);
    state.assign(this->bad.begin(), this->bad.end());
    restarts.assign(nb, 0);
    WF_TRY(start_cg(c, B, st));
    phase = 1;
    return WF_OK;
  }
  // r = C F(rhs) for every system; p = 0; reset the recurrences of the running systems
  wf_status start_cg(Ctx& c, const double* rhs, cudaStream_t st) {
    const size_t SPEC = SP::SPEC;
    SP::zfwd(c, nb, rhs, T, tw, nullptr, st);
    SP::ypass(c, nb, T, tw, nullptr, -1, st);
    SP::template xmul<true, false, true>(c, nb, T, rh, ct, tw, part, nullptr, st);
    const Bat b = SP::bat();
    c.launch("fin", 0, st, [&] { k_fin_init<<<nb, 1024, 0, st>>>(part, SP::GXF, sc, b); });
    WF_CUDA(cudaMemsetAsync(P0, 0, nb * SPEC * sizeof(ST), st));
    WF_CUDA(cudaMemsetAsync(P1, 0, nb * SPEC * sizeof(ST), st));
    WF_CUDA(cudaGetLastError());
    return WF_OK;
  }
  wf_status block(Ctx& c, cudaStream_t st) {
    return this->run_block(c, st, [&](cudaStream_t s2) {
      for (int i = 0; i < check_every<N>(); ++i)
        SP::iteration(c, nb, rh, P0, P1, xh, T, D, ct, mt, unit_m, tw, part, sc, inv_vc, s2);
    });
  }
  wf_status enqueue(Ctx& c, cudaStream_t st) override {
    if (phase == 1) {
      WF_TRY(block(c, st));
    } else if (phase == 2) {
      const Bat b = SP::bat();
      c.launch("axpy", 3 * SP::BS * nb, st,
               [&] { k_axpy_final<<<dim3(152 * 4, nb), 256, 0, st>>>(xh, P0, P1, SP::SPEC, sc, b); });
      SP::template xmul<false, true, false>(c, nb, xh, T, ct, tw, part, nullptr, st);
      SP::ypass(c, nb, T, tw, nullptr, +1, st);
      SP::template zinv<ZI_STORE>(c, nb, T, S, nullptr, nullptr, nullptr, inv_vc, tw, part, nullptr, st);
      // residual b - A s
      SP::zfwd(c, nb, S, T, tw, nullptr, st);
      SP::ypass(c, nb, T, tw, nullptr, -1, st);
      SP::fmul(c, nb, T, T2, stab, &sc->texp, this->kScalInts, st);
      SP::ypass(c, nb, T2, tw, nullptr, +1, st);
      SP::template zinv<ZI_RESID>(c, nb, T2, RES, S, W, B, inv_vc, tw, part, sc, st);
      c.launch("fin", 0, st, [&] { k_fin_sum<<<nb, 1024, 0, st>>>(part, SP::GZI, 0, sc, b); });
    } else if (phase == 3) {
      WF_TRY(this->push_scalars(st));
      WF_TRY(start_cg(c, RES, st));
      phase = 1;
      WF_TRY(block(c, st));
    }
    WF_CUDA(cudaGetLastError());
    return this->pull_scalars(st);
  }
  wf_status advance(Ctx&) override {
    this->read_scalars();
    if (phase == 1) {
      if (this->all_done()) phase = 2;
      return WF_OK;
    }
    if (phase == 2) {
      bool any = false;
      for (int m = 0; m < nb; ++m) {
        if (state[m]) {
          h[m].done = 4;
          continue;
        }
        rel[m] = bb0[m] > 0 ? std::sqrt(h[m].aux[0] / bb0[m]) : 0.0;
        wf_status st = WF_OK;
        bool fin = true;
        if (bb0[m] == 0.0 || rel[m] <= sys[m]->opts.tol) st = WF_OK;
        else if (h[m].done == 3) st = WF_ERR_BREAKDOWN;
        else if (h[m].iter >= sys[m]->opts.max_iter || restarts[m] >= 8) st = WF_ERR_NOT_CONVERGED;
        else fin = false;
        if (fin) {
          state[m] = 1;
          h[m].done = 4;
          if (info[m]) *info[m] = wf_solve_info{h[m].iter, restarts[m], rel[m], sys[m]->nbar, st};
        } else {
          restarts[m] += 1;
          h[m].done = 0;
          any = true;
        }
      }
      phase = any ? 3 : 9;
    }
    return WF_OK;
  }
  bool done() const override { return phase == 9; }
  wf_status finish(Ctx&, cudaStream_t st) override {
    for (int m = 0; m < nb; ++m)
      WF_CUDA(cudaMemcpyAsync(sys[m]->s_out, S + m * SP::V, SP::V * sizeof(double), cudaMemcpyDefault, st));
    return WF_OK;
  }
};

// ------------------------------------------------------------------------------------------
// Mixed group: outer FP64 refinement x += e, inner CG on A e = res in FP32 spectra.
// Phases: 0 inner start, 1 CG loop, 2 accumulate + FP64 residual, 9 done.
// ------------------------------------------------------------------------------------------
template <int N>
struct GroupMixed : GroupCommon<N> {
  using SF = Spec<float, N>;
  using SD = Spec<FP64Arith, N>;
  using Base = GroupCommon<N>;
  using Base::nb; using Base::sys; using Base::info; using Base::key; using Base::W; using Base::B;
  using Base::S; using Base::RES; using Base::part; using Base::sc; using Base::tw; using Base::h;
  using Base::phase; using Base::inv_vc; using Base::bb0; using Base::rel; using Base::state;
  float2 *xh, *rh, *P0, *P1, *T;
  float* D;
  double2 *T64, *T64b;
  const float2* tw32 = nullptr;  // FP32 copy of the twiddle table for the FP32 passes
  float *ct, *mt;
  double* stab;
  std::vector<int> outer, iters;
  std::vector<int> texp;  // per system: power of two of the prior table's digits
  std::vector<int> noco;  // per system: inner solves without the coarse space after a failed one
  bool unit_m = true;
  static constexpr int NPART = SF::NPART > SD::NPART ? SF::NPART : SD::NPART;
  // coarse space of a deflated group (K > 0; every system of the group has the same K)
  int K = 0, nh = 0, ncp = 0;
  int4* dmodes = nullptr;
  float *Einv = nullptr, *gco = nullptr, *rco = nullptr, *Pb = nullptr, *Rp = nullptr, *Cp = nullptr;
  float2 *Gz = nullptr, *Gy = nullptr, *rsave = nullptr, *DH = nullptr;
  double *dpart = nullptr, *normp = nullptr;  // normp: per-CTA row-sum maxima of E and E^-1
  int* doff = nullptr;  // per system: 1 = the coarse block failed the condition guard (plain CG)
  size_t gzs = 0, gys = 0;

  wf_status prepare_begin(Ctx& c, cudaStream_t st) override {
    nb = (int)sys.size();
    K = sys[0]->opts.deflate;
    // groups of one size with different coarse radii run side by side: their workspaces differ by K
    key = this->tag + "mix_" + std::to_string(N) + "_" + (K > 0 ? "k" + std::to_string(K) + "_" : std::string());
    int* err;
    WF_TRY(c.err_word(&err));
    WF_CUDA(SF::attrs());
    WF_CUDA(SD::attrs());
    const size_t SPEC = SF::SPEC, V = SF::V;
    WF_TRY(c.tw(N, &tw));
    WF_TRY(c.tw32(N, &tw32));
    WF_TRY(c.fix_tables(N));
    const char* nm[5] = {"x", "r", "p0", "p1", "T"};
    float2** ptr[5] = {&xh, &rh, &P0, &P1, &T};
    for (int i = 0; i < 5; ++i) WF_TRY(c.get(key + nm[i], nb * SPEC * sizeof(float2), (void**)ptr[i]));
    WF_TRY(c.get(key + "D", nb * V * sizeof(float), (void**)&D));
    WF_TRY(c.get(key + "T64", nb * SPEC * sizeof(double2), (void**)&T64));
    WF_TRY(c.get(key + "T64b", nb * SPEC * sizeof(double2), (void**)&T64b));
    WF_TRY(c.get(key + "W", nb * V * sizeof(double), (void**)&W));
    WF_TRY(c.get(key + "B", nb * V * sizeof(double), (void**)&B));
    WF_TRY(c.get(key + "S", nb * V * sizeof(double), (void**)&S));
    WF_TRY(c.get(key + "RES", nb * V * sizeof(double), (void**)&RES));
    WF_TRY(c.get(key + "part", (size_t)nb * NPART * sizeof(double), (void**)&part));
    WF_TRY(c.get(key + "sc", nb * sizeof(CgScal), (void**)&sc));
    WF_TRY(c.get_pinned(key + "hsc", nb * sizeof(CgScal), (void**)&this->hsc));
    for (int m = 0; m < nb; ++m) {
      WF_CUDA(cudaMemcpyAsync(W + m * V, sys[m]->w, V * sizeof(double), cudaMemcpyDefault, st));
      WF_CUDA(cudaMemcpyAsync(B + m * V, sys[m]->b, V * sizeof(double), cudaMemcpyDefault, st));
    }
    if (K > 0) WF_TRY(defl_alloc(c, st));
    return group_sums_begin<N>(c, *this, NPART, st);
  }
  // the coarse-space buffers and the mode table
  wf_status defl_alloc(Ctx& c, cudaStream_t st) {
    const std::vector<int4> modes = deflation_modes(K);
    nh = (int)modes.size();
    ncp = deflation_ncp(K);
    const size_t C = 4 * K + 1;
    gzs = (size_t)N * N * (K + 1);
    gys = (size_t)(2 * K + 1) * (K + 1) * N;
    const std::string dk = key + "d" + std::to_string(K) + "_";
    WF_TRY(c.get(dk + "E", (size_t)nb * ncp * ncp * sizeof(float), (void**)&Einv));
    WF_TRY(c.get(dk + "gco", (size_t)nb * ncp * sizeof(float), (void**)&gco));
    WF_TRY(c.get(dk + "rco", (size_t)nb * ncp * sizeof(float), (void**)&rco));
    WF_TRY(c.get(dk + "P", (size_t)nb * 2 * kDeflTile * kDeflTile * sizeof(float), (void**)&Pb));
    WF_TRY(c.get(dk + "Rp", (size_t)nb * kDeflTile * ncp * sizeof(float), (void**)&Rp));
    WF_TRY(c.get(dk + "Cp", (size_t)nb * ncp * kDeflTile * sizeof(float), (void**)&Cp));
    WF_TRY(c.get(dk + "Gz", (size_t)nb * gzs * sizeof(float2), (void**)&Gz));
    WF_TRY(c.get(dk + "Gy", (size_t)nb * gys * sizeof(float2), (void**)&Gy));
    WF_TRY(c.get(dk + "rsave", (size_t)nb * (2 * nh + 1) * sizeof(float2), (void**)&rsave));
    WF_TRY(c.get(dk + "DH", (size_t)nb * C * C * C * sizeof(float2), (void**)&DH));
    WF_TRY(c.get(dk + "dpart", (size_t)nb * (nh + 1) * sizeof(double), (void**)&dpart));
    WF_TRY(c.get(dk + "normp", (size_t)nb * 2 * (ncp / 8) * sizeof(double), (void**)&normp));
    WF_TRY(c.get(dk + "doff", (size_t)nb * sizeof(int), (void**)&doff));
    WF_TRY(c.get(dk + "modes", modes.size() * sizeof(int4), (void**)&dmodes));
    int4* hm;
    WF_TRY(c.get_pinned(dk + "hmodes", modes.size() * sizeof(int4), (void**)&hm));
    std::copy(modes.begin(), modes.end(), hm);
    WF_CUDA(cudaMemcpyAsync(dmodes, hm, modes.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
    WF_CUDA(cudaMemsetAsync(gco, 0, (size_t)nb * ncp * sizeof(float), st));
    WF_CUDA(cudaMemsetAsync(rco, 0, (size_t)nb * ncp * sizeof(float), st));
    return WF_OK;
  }
  // E^-1 of every system: the transform of w (FP32 passes, P0 as scratch), Dh at the differences
  // of coarse modes, the Galerkin block, and its block Gauss-Jordan exchange
  wf_status defl_setup(Ctx& c, cudaStream_t st) {
    const Bat bf = SF::bat();
    std::vector<double> ones((size_t)nb * SF::TAB, 1.0);
    float* tone;
    WF_TRY(upload_tables<float>(c, key + "t1", ones, &tone, st));
    SF::zfwd(c, nb, W, T, tw32, nullptr, st);
    SF::ypass(c, nb, T, tw32, nullptr, -1, st);
    SF::template xmul<true, false, true>(c, nb, T, P0, tone, tw32, part, nullptr, st);
    const int C = 4 * K + 1;
    c.launch("defl_dh", 0, st, [&] {
      k_dh_gather<float, N><<<dim3((C * C * C + 255) / 256, nb), 256, 0, st>>>(P0, DH, K, inv_vc, sc, bf);
    });
    c.launch("defl_E", 0, st, [&] {
      k_ebuild<float><<<dim3(ncp / 16, ncp / 16, nb), dim3(16, 16), 0, st>>>(DH, ct, mt, dmodes, nh, ncp, K, Einv,
                                                                            SF::TAB);
    });
    const int nbk = ncp / kDeflTile;
    double* pe = normp;
    double* pi = normp + (size_t)nb * (ncp / 8);
    c.launch("defl_norm", 0, st, [&] { k_defl_rownorm<<<dim3(ncp / 8, nb), 256, 0, st>>>(Einv, ncp, pe); });
    c.launch("gj_pivot", 0, st, [&] { k_gj_pivot<<<dim3(1, 1, nb), 64, 0, st>>>(Einv, Pb, ncp); });
    for (int kb = 0; kb < nbk; ++kb) {
      c.launch("gj_panel", 0, st, [&] { k_gj_panel<<<dim3(nbk, 1, nb), 64, 0, st>>>(Einv, Pb, Rp, Cp, ncp, kb); });
      c.launch("gj_update", 0, st, [&] {
        k_gj_update<<<dim3(nbk / 2, nbk / 2, nb), 256, kUpdSmem, st>>>(Einv, Pb, Rp, Cp, ncp, kb);
      });
    }
    c.launch("defl_norm", 0, st, [&] { k_defl_rownorm<<<dim3(ncp / 8, nb), 256, 0, st>>>(Einv, ncp, pi); });
    c.launch("defl_norm", 0, st, [&] { k_defl_guard<<<nb, 256, 0, st>>>(pe, pi, ncp, doff); });
    WF_CUDA(cudaGetLastError());
    return WF_OK;
  }
  // coordinates of A' r - r and of r, and r -= Z E^-1 g kept aside (MODE 1); or the start vector
  // Z E^-1 Z^T r into `out` (MODE 0)
  template <int MODE>
  void defl_project(Ctx& c, float2* out, cudaStream_t st, int n3 = 0) {
    const Bat bf = SF::bat();
    const int gw = (nh + 1 + 7) / 8;
    if constexpr (MODE == 1) {
      c.launch("defl_xr", 2 * SF::BS * nb, st,
               [&] { Ctx::chain(k_xcr<float, N, 32>, SF::gxy(nb), SF::NTx, SF::SMxy, st, rh, T, ct, tw32, sc, bf); });
      SF::ypass(c, nb, T, tw32, sc, +1, st);
      c.launch("defl_z", (SF::BS + 4 * SF::BV) * nb, st, [&] {
        Ctx::chain(k_zcoarse<float, N>, SF::gz(nb), SF::NTz, SF::SMz, st, T, D, tw32, Gz, K, sc, bf, gzs);
      });
      const size_t ysm = ((size_t)N * (K + 1) + N) * sizeof(float2);
      c.launch("defl_y", 8.0 * gzs * nb, st, [&] {
        Ctx::chain(k_ycoarse<float, N>, dim3(N + (n3 > 0), nb), 256, ysm, st, Gz, tw32, Gy, K, sc, gzs, gys, bf, part, n3,
                   inv_vc);
      });
    }
    c.launch("defl_x", 8.0 * gys * nb, st, [&] {
      Ctx::chain(k_xcoarse<float, N, MODE>, dim3(gw, nb), 256, 0, st, Gy, rh, ct, mt, tw32, dmodes, nh, K, gco, rco, sc,
                 bf, gys, ncp);
    });
    c.launch("defl_mu", 4.0 * ncp * ncp * nb, st, [&] {
      Ctx::chain(k_defl_mu<float, N, MODE>, dim3(gw, nb), 256, ncp * sizeof(float), st, Einv, gco, rco, dmodes, nh, ncp,
                 out, rsave, dpart, sc, bf, doff);
    });
  }
  // one deflated inner iteration: p = (r - Z mu) + beta p with mu from the coarse projection.  n3 > 0: beta and the stop
  // test of the iteration before are still to be taken, by the coarse y stage; the same is left to the caller here
  // unless this is the last one before the host looks (the return value).
  int defl_iteration(Ctx& c, cudaStream_t st, int n3, bool last) {
    defl_project<1>(c, rh, st, n3);
    YFin fin;
    fin.nh = nh;
    fin.r = rh;
    fin.rsave = rsave;
    fin.modes = dmodes;
    n3 = SF::iteration(c, nb, rh, P0, P1, xh, T, D, ct, mt, unit_m, tw32, part, sc, inv_vc, st, nullptr, fin, last);
    return last ? 0 : n3;
  }
  wf_status prepare_end(Ctx& c, cudaStream_t st) override {
    const size_t V = SF::V;
    group_sums_end<N>(*this);
    const int TAB = SF::TAB;
    std::vector<double> vc((size_t)nb * TAB), vm((size_t)nb * TAB), vs((size_t)nb * TAB);
    unit_m = true;
    for (int m = 0; m < nb; ++m) {
      const bool pre = sys[m]->opts.precond != 0;
      unit_m = unit_m && pre;
      const double c0 = 1.0 / std::sqrt(sys[m]->nbar * this->sumw[m] * inv_vc);
      make_tables(sys[m]->sinv, pre, c0, vc.data() + (size_t)m * TAB, vm.data() + (size_t)m * TAB);
      std::copy(sys[m]->sinv.begin(), sys[m]->sinv.end(), vs.begin() + (size_t)m * TAB);
    }
    WF_TRY(upload_tables<float>(c, key + "tc", vc, &ct, st));
    WF_TRY(upload_tables<float>(c, key + "tm", vm, &mt, st));
    WF_TRY(upload_tables<double>(c, key + "ts", vs, &stab, st));
    h.assign(nb, CgScal{});
    texp.resize(nb);
    for (int m = 0; m < nb; ++m) {
      h[m].nbar = sys[m]->nbar;
      h[m].texp = texp[m] = table_exp(sys[m]->sinv.data(), TAB);
    }
    WF_TRY(this->push_scalars(st));
    if constexpr (!SD::BUTTERFLY_RESID) this->table_digits(c, stab, st);
    c.launch("make_D", 12.0 * V * nb, st, [&] { k_make_D<float><<<dim3(152 * 4, nb), 256, 0, st>>>(W, D, sc, inv_vc, V); });
    if (K > 0) WF_TRY(defl_setup(c, st));
    // x = 0 (accumulated in S), res = b
    WF_CUDA(cudaMemsetAsync(S, 0, nb * V * sizeof(double), st));
    WF_CUDA(cudaMemcpyAsync(RES, B, nb * V * sizeof(double), cudaMemcpyDeviceToDevice, st));
    rel.assign(nb, 1.0);
    state.assign(this->bad.begin(), this->bad.end());
    outer.assign(nb, 0);
    iters.assign(nb, 0);
    noco.assign(nb, 0);
    for (int m = 0; m < nb; ++m)
      if (bb0[m] == 0.0 && !state[m]) {
        state[m] = 1;
        rel[m] = 0.0;
        if (info[m]) *info[m] = wf_solve_info{0, 0, 0.0, sys[m]->nbar, WF_OK};
      }
    phase = 0;
    return WF_OK;
  }
  wf_status enqueue(Ctx& c, cudaStream_t st) override {
    const Bat bf = SF::bat();
    if (phase == 0) {
      // Each inner solve aims at the remaining reduction (kInnerMargin of it) but at most
      // inner_tol (1e-4 by default) per step, so at least two FP64 refinement steps run for
      // tol <= 1e-6: the second removes the FP32 rounding error the first leaves in the
      // low-eigenvalue directions (at 512^3 a single step to 1e-6 saves ~6% of the iterations but
      // leaves the solution 3.6e-5 from the converged one, two steps 5e-7).
      const double inner_tol_def = 1e-4;
      for (int m = 0; m < nb; ++m) {
        CgScal z{};
        z.nbar = sys[m]->nbar;
        z.texp = texp[m];
        if (state[m]) {
          z.done = 4;
        } else {
          const double itol = sys[m]->opts.inner_tol > 0.0 ? sys[m]->opts.inner_tol : inner_tol_def;
          const double target = std::max(itol, kInnerMargin * sys[m]->opts.tol / rel[m]);
          z.tol2 = target * target;
          z.bb = rel[m] * rel[m] * bb0[m];
          z.max_iter = std::max(1, sys[m]->opts.max_iter - iters[m]);
          if (K > 0 && !noco[m]) z.max_iter = std::min(z.max_iter, kDeflInnerCap);
          z.noco = noco[m];
          outer[m] += 1;
        }
        h[m] = z;
      }
      WF_TRY(this->push_scalars(st));
      const size_t SPEC = SF::SPEC;
      SF::zfwd(c, nb, RES, T, tw32, nullptr, st);
      SF::ypass(c, nb, T, tw32, nullptr, -1, st);
      SF::template xmul<true, false, true>(c, nb, T, rh, ct, tw32, part, nullptr, st);
      c.launch("fin", 0, st, [&] { k_fin_init<<<nb, 1024, 0, st>>>(part, SF::GXY, sc, bf); });
      WF_CUDA(cudaMemsetAsync(P0, 0, nb * SPEC * sizeof(float2), st));
      WF_CUDA(cudaMemsetAsync(P1, 0, nb * SPEC * sizeof(float2), st));
      WF_CUDA(cudaMemsetAsync(xh, 0, nb * SPEC * sizeof(float2), st));
      if (K > 0) {
        // the start step of the two-level form: p = Z E^-1 Z^T r (in the FP64 scratch spectrum),
        // taken with alpha = 1 so that x = Z E^-1 Z^T b and Z^T r = 0 afterwards
        float2* Rc = reinterpret_cast<float2*>(T64);
        WF_CUDA(cudaMemsetAsync(Rc, 0, nb * SPEC * sizeof(float2), st));
        c.launch("fin", 0, st, [&] { k_defl_arm<<<nb, 32, 0, st>>>(sc); });
        defl_project<0>(c, Rc, st);
        SF::iteration(c, nb, rh, P0, P1, xh, T, D, ct, mt, unit_m, tw32, part, sc, inv_vc, st, Rc);
      }
      phase = 1;
    }
    if (phase == 1) {
      WF_TRY(this->run_block(c, st, [&](cudaStream_t s2) {
        int n3 = 0;
        for (int i = 0; i < check_every<N>(); ++i) {
          if (K > 0) n3 = defl_iteration(c, s2, n3, i == check_every<N>() - 1);
          else SF::iteration(c, nb, rh, P0, P1, xh, T, D, ct, mt, unit_m, tw32, part, sc, inv_vc, s2);
        }
      }));
    } else if (phase == 2) {
      c.launch("axpy", 3 * SF::BS * nb, st,
               [&] { k_axpy_final<<<dim3(152 * 4, nb), 256, 0, st>>>(xh, P0, P1, SF::SPEC, sc, bf); });
      // x += C e (FP32 transform, FP64 accumulation) for the systems that ran
      SF::template xmul<false, true, false>(c, nb, xh, T, ct, tw32, part, nullptr, st);
      SF::ypass(c, nb, T, tw32, nullptr, +1, st);
      SF::template zinv<ZI_ACCUM>(c, nb, T, S, nullptr, nullptr, nullptr, inv_vc, tw32, part, sc, st);
      // FP64 residual res = b - A x
      const int np = SD::resid(c, nb, S, W, B, RES, T64, T64b, stab, &sc->texp, this->kScalInts, inv_vc, tw, part, sc, st);
      const Bat bd = SD::bat();
      c.launch("fin", 0, st, [&] { k_fin_sum<<<nb, 1024, 0, st>>>(part, np, 0, sc, bd); });
    }
    WF_CUDA(cudaGetLastError());
    return this->pull_scalars(st);
  }
  wf_status advance(Ctx&) override {
    this->read_scalars();
    if (phase == 1) {
      if (this->all_done()) phase = 2;
      return WF_OK;
    }
    if (phase == 2) {
      bool any = false;
      for (int m = 0; m < nb; ++m) {
        if (state[m]) continue;
        iters[m] += h[m].iter;
        const double rn = std::sqrt(h[m].aux[0] / bb0[m]);
        const bool broke = h[m].done == 3 && !(rn < rel[m]);
        // a deflated inner solve that broke down or reached kDeflInnerCap hands the system to plain
        // CG from the next refinement step on (its FP64 residual restarts the inner solve)
        const bool defl_failed = K > 0 && !noco[m] && std::isfinite(rn) &&
                                 (h[m].done == 3 || (h[m].done == 2 && h[m].iter >= kDeflInnerCap));
        rel[m] = rn;
        wf_status st = WF_OK;
        bool fin = true;
        if (rel[m] <= sys[m]->opts.tol) st = WF_OK;
        else if (defl_failed && outer[m] < 12 && iters[m] < sys[m]->opts.max_iter) {
          noco[m] = 1;
          fin = false;
        } else if (broke) st = WF_ERR_BREAKDOWN;
        else if (outer[m] >= 12 || iters[m] >= sys[m]->opts.max_iter) st = WF_ERR_NOT_CONVERGED;
        else fin = false;
        if (fin) {
          state[m] = 1;
          if (info[m]) *info[m] = wf_solve_info{iters[m], outer[m], rel[m], sys[m]->nbar, st};
        } else {
          any = true;
        }
      }
      phase = any ? 0 : 9;
    }
    return WF_OK;
  }
  bool done() const override { return phase == 9; }
  wf_status finish(Ctx&, cudaStream_t st) override {
    for (int m = 0; m < nb; ++m)
      WF_CUDA(cudaMemcpyAsync(sys[m]->s_out, S + m * SF::V, SF::V * sizeof(double), cudaMemcpyDefault, st));
    return WF_OK;
  }
};

// out = F^-1 [g(|m|^2) F in] for one FP64 field, with the multiplier given as a table over
// n2 = |m|^2 (3 (N/2)^2 + 1 entries): the Gaussian smoothing of Sec. 4.1 and the deconvolution
// B^-1 Z^-1 of Eq. eq:DEC.  The x pass applies the table as it applies the prior; the transforms
// are the solver's FP64 passes.  in may equal out.
template <int N>
wf_status fourier_multiply_n(Ctx& c, const double* in, double* out, const std::vector<double>& table, double kf,
                             double r_s, cudaStream_t st) {
  using SD = Spec<FP64Arith, N>;
  const bool gauss = table.empty();
  if (!gauss && (int)table.size() != SD::TAB) return WF_ERR_ARG;
  int* err;
  WF_TRY(c.err_word(&err));
  WF_CUDA(SD::attrs());
  WF_TRY(c.fix_tables(N));
  double2 *T, *T2;
  int *exps, *hexp;
  WF_TRY(c.get("sm_T", SD::SPEC * sizeof(double2), (void**)&T));
  WF_TRY(c.get("sm_T2", SD::SPEC * sizeof(double2), (void**)&T2));
  WF_TRY(c.get("sm_e", sizeof(int), (void**)&exps));
  WF_TRY(c.get_pinned("sm_eh", sizeof(int), (void**)&hexp));
  double* gt;
  if (gauss) {
    WF_TRY(c.get("sm_g", SD::TAB * sizeof(double), (void**)&gt));
    c.launch("tables", 0, st, [&] { k_gauss_table<<<(SD::TAB + 255) / 256, 256, 0, st>>>(gt, SD::TAB, kf, r_s); });
    // the largest entry is 1; an exponent's infinity times 0 makes the first or the last one a NaN
    const double h = -0.5 * kf * kf;
    *hexp = std::isnan(h * 0.0 * r_s * r_s) || std::isnan(h * (double)(SD::TAB - 1) * r_s * r_s) ? kFxNanTab : 1;
  } else {
    WF_TRY(upload_tables<double>(c, "sm_g", table, &gt, st));
    *hexp = table_exp(table.data(), table.size());
  }
  WF_CUDA(cudaMemcpyAsync(exps, hexp, sizeof(int), cudaMemcpyHostToDevice, st));
  c.launch("tables", 0, st, [&] { k_table_digits<<<dim3((SD::TAB + 255) / 256, 1), 256, 0, st>>>(gt, SD::TAB, exps, 1); });
  SD::zfwd(c, 1, in, T, nullptr, nullptr, st);
  using Y = typename SD::template YFix<FxWide>;  // a caller's field may have any magnitude
  Y::run(c, 1, T, nullptr, nullptr, -1, st, YFin{});
  SD::fmul(c, 1, T, T2, gt, exps, 1, st);
  Y::run(c, 1, T2, nullptr, nullptr, +1, st, YFin{});
  SD::template zinv<ZI_STORE>(c, 1, T2, out, nullptr, nullptr, nullptr, 1.0 / (double)SD::V, nullptr, nullptr, nullptr,
                              st);
  WF_CUDA(cudaGetLastError());
  WF_CUDA(cudaStreamSynchronize(st));
  return c.check_device_errors();
}

// ---- autotuner: time each launch variant of a pass on a working set larger than L2 ----------
template <class SP, class V>
wf_status tune_pass(Ctx& c, const char* pass, const std::vector<V>& vs, typename SP::ST* buf, int nb,
                    const typename SP::ST* tw, cudaStream_t st, std::string& report) {
  const std::string key = SP::tune_key(pass);
  char head[160];
  std::snprintf(head, sizeof head, "{\"pass\": \"%s\", \"systems\": %d, \"variants\": [", key.c_str(), nb);
  report += head;
  cudaEvent_t a, b;
  WF_CUDA(cudaEventCreate(&a));
  WF_CUDA(cudaEventCreate(&b));
  int best = 0;
  float best_ms = 1e30f;
  const bool prof = c.prof.on;
  c.prof.on = false;  // the tuner's launches are not part of a profile
  wf_status status = WF_OK;
  for (size_t i = 0; i < vs.size() && status == WF_OK; ++i) {
    constexpr int kWarm = 2, kRuns = 6;
    for (int r = 0; r < kWarm; ++r) vs[i].run(c, nb, buf, tw, nullptr, -1, st);
    cudaEventRecord(a, st);
    for (int r = 0; r < kRuns; ++r) vs[i].run(c, nb, buf, tw, nullptr, r & 1 ? +1 : -1, st);
    cudaEventRecord(b, st);
    cudaError_t e = cudaEventSynchronize(b);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, a, b);
    if (e != cudaSuccess) {
      set_last_error("autotune timing", e);
      status = WF_ERR_CUDA;
      break;
    }
    ms /= kRuns;
    char item[128];
    std::snprintf(item, sizeof item, "%s{\"name\": \"%s\", \"ms\": %.5f}", i ? ", " : "", vs[i].name, ms);
    report += item;
    if (ms < best_ms) {
      best_ms = ms;
      best = (int)i;
    }
  }
  c.prof.on = prof;
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  WF_TRY(status);
  WF_TRY(c.check_device_errors());
  c.tuned[key] = best;
  char tail[96];
  std::snprintf(tail, sizeof tail, "], \"chosen\": \"%s\"}", vs[best].name);
  report += tail;
  return WF_OK;
}

template <class SP>
wf_status tune_spec(Ctx& c, std::string& report) {
  using ST = typename SP::ST;
  int* err;
  WF_TRY(c.err_word(&err));
  WF_CUDA(SP::attrs());
  WF_TRY(c.fix_tables(SP::NH * 2));
  const ST* tw;
  if constexpr (sizeof(typename SP::SS) == 8) {
    WF_TRY(c.tw(SP::NH * 2, &tw));
  } else {
    WF_TRY(c.tw32(SP::NH * 2, &tw));
  }
  // enough systems that the working set (read and written once per pass) is at least 256 MB,
  // so that the passes stream from HBM as they do in a large solve or a batch
  const double spec_bytes = (double)SP::SPEC * sizeof(ST);
  int nb = (int)std::ceil((256.0 * (1 << 20)) / spec_bytes);
  nb = std::max(1, std::min(nb, 64));
  ST* buf;
  WF_TRY(c.get("tune_spec", (size_t)nb * SP::SPEC * sizeof(ST), (void**)&buf));
  cudaStream_t st;
  WF_TRY(c.stream(0, &st));
  WF_CUDA(cudaMemsetAsync(buf, 0, (size_t)nb * SP::SPEC * sizeof(ST), st));
  WF_TRY(tune_pass<SP>(c, "ypass", SP::yvariants(), buf, nb, tw, st, report));
  WF_CUDA(cudaStreamSynchronize(st));
  c.release_prefix("tune_spec");
  // the CG x passes: five spectra per system, scalars of running systems, unit tables
  using SS = typename SP::SS;
  const size_t SPEC = SP::SPEC;
  ST* xb;
  SS* tab;
  double* part;
  CgScal* sc;
  WF_TRY(c.get("tune_x", (size_t)5 * nb * SPEC * sizeof(ST), (void**)&xb));
  const size_t ntab = (size_t)nb * SP::TAB;
  WF_TRY(c.get("tune_xtab", ntab * sizeof(SS), (void**)&tab));
  WF_TRY(c.get("tune_xpart", (size_t)nb * SP::NPART * sizeof(double), (void**)&part));
  WF_TRY(c.get("tune_xsc", (size_t)nb * sizeof(CgScal), (void**)&sc));
  WF_CUDA(cudaMemsetAsync(xb, 0, (size_t)5 * nb * SPEC * sizeof(ST), st));
  WF_CUDA(cudaMemsetAsync(sc, 0, (size_t)nb * sizeof(CgScal), st));
  {
    std::vector<SS> ones(ntab, (SS)1);
    WF_CUDA(cudaMemcpyAsync(tab, ones.data(), ones.size() * sizeof(SS), cudaMemcpyHostToDevice, st));
    WF_CUDA(cudaStreamSynchronize(st));
  }
  ST *r = xb, *P0 = xb + nb * SPEC, *P1 = xb + 2 * nb * SPEC, *x = xb + 3 * nb * SPEC, *T = xb + 4 * nb * SPEC;
  struct XRun {
    const typename SP::XVariant* v;
    bool inv;
    const char* name;
    void run(Ctx& c, int nb, cudaStream_t st, ST* r, ST* P0, ST* P1, ST* x, ST* T, const SS* tab, const ST* tw,
             double* part, CgScal* sc, int, int) const {
      if (inv) v->xinv(c, nb, r, P0, P1, x, T, tab, tab, true, tw, part, sc, st);
      else v->xupd(c, nb, T, r, P0, P1, tab, tab, true, tw, part, sc, st);
    }
  };
  for (int inv = 1; inv >= 0; --inv) {
    std::vector<XRun> runs;
    for (const auto& v : SP::xvariants()) runs.push_back(XRun{&v, inv == 1, v.name});
    struct Adapter {
      const XRun* x;
      ST *r, *P0, *P1, *xx, *T;
      const SS* tab;
      double* part;
      CgScal* sc;
      const char* name;
      void run(Ctx& c, int nb, ST*, const ST* tw, const CgScal*, int, cudaStream_t st) const {
        x->run(c, nb, st, r, P0, P1, xx, T, tab, tw, part, sc, 0, 0);
      }
    };
    std::vector<Adapter> ad;
    for (const auto& rr : runs) ad.push_back(Adapter{&rr, r, P0, P1, x, T, tab, part, sc, rr.name});
    report += ", ";
    WF_TRY(tune_pass<SP>(c, inv ? "xinv" : "xupd", ad, r, nb, tw, st, report));
  }
  {  // the z turn: T and D (FP32/FP64 real field, one spectrum's bytes or half) from the scratch
    struct ZAdapter {
      const typename SP::ZVariant* v;
      SS* D;
      double* part;
      CgScal* sc;
      const char* name;
      void run(Ctx& c, int nb, ST* buf, const ST* tw, const CgScal*, int, cudaStream_t st) const {
        v->run(c, nb, buf, D, tw, part, sc, st);
      }
    };
    std::vector<ZAdapter> za;
    SS* D = reinterpret_cast<SS*>(x);  // the x buffer holds nb fields of V reals (zeroed)
    for (const auto& v : SP::zvariants()) za.push_back(ZAdapter{&v, D, part, sc, v.name});
    report += ", ";
    WF_TRY(tune_pass<SP>(c, "zturn", za, T, nb, tw, st, report));
  }
  WF_CUDA(cudaStreamSynchronize(st));
  c.release_prefix("tune_x");
  return WF_OK;
}

template <int N>
wf_status autotune_n(Ctx& c, int prec, std::string& report) {
  if (prec == WF_MIXED) return tune_spec<Spec<float, N>>(c, report);
  return tune_spec<Spec<FP64Arith, N>>(c, report);
}

template <int N>
Group* make_group(int prec) {
  if (prec == WF_MIXED) return new GroupMixed<N>();
  return new GroupFP64<FP64Arith, N>();
}

}  // namespace wf
