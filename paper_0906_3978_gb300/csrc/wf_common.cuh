// wf_common.cuh -- arithmetic types, complex helpers and reductions shared by the kernels.
//
// Two real types carry the spectral arithmetic: double (the 1/64-rate unit) and float; FP64-stored fields also go
// through 64-bit fixed point (wf_fix.cuh).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#define WF_HD __host__ __device__ __forceinline__
#define WF_D __device__ __forceinline__

// s + e = a + b exactly (Knuth two-sum, no magnitude assumption)
WF_D void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// Ask L2 to fetch [p, p + bytes) from HBM ahead of its use (a bulk prefetch: no registers or
// shared memory held, no completion to wait for).  p and bytes must be multiples of 16.
WF_D void prefetch_l2(const void* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// ------------------------------------------------------------------------------------------
// real-type traits: constants and conversion to/from the FP64 / FP32 storage types
// ------------------------------------------------------------------------------------------
template <class R> struct RT;
template <> struct RT<double> {
  WF_HD static double c(double v) { return v; }
  WF_D static double from_d(double v) { return v; }
  WF_D static double to_d(double v) { return v; }
  WF_D static double from_f(float v) { return (double)v; }
  WF_D static float to_f(double v) { return (float)v; }
};
template <> struct RT<float> {
  WF_HD static float c(double v) { return (float)v; }
  WF_D static float from_d(double v) { return __double2float_rn(v); }
  WF_D static double to_d(float v) { return (double)v; }
  WF_D static float from_f(float v) { return v; }
  WF_D static float to_f(float v) { return v; }
};
// ------------------------------------------------------------------------------------------
// complex over a real type
// ------------------------------------------------------------------------------------------
template <class R> struct __align__(2 * sizeof(R)) cx {
  R x, y;
};
template <class R> WF_D cx<R> operator+(cx<R> a, cx<R> b) { return cx<R>{a.x + b.x, a.y + b.y}; }
template <class R> WF_D cx<R> operator-(cx<R> a, cx<R> b) { return cx<R>{a.x - b.x, a.y - b.y}; }
template <class R> WF_D cx<R> operator*(cx<R> a, cx<R> b) {
  return cx<R>{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <class R> WF_D cx<R> scale(cx<R> a, R s) { return cx<R>{a.x * s, a.y * s}; }
template <class R> WF_D cx<R> conj(cx<R> a) { return cx<R>{a.x, -a.y}; }
template <class R> WF_D cx<R> mul_i(cx<R> a) { return cx<R>{-a.y, a.x}; }      // a * i
template <class R> WF_D cx<R> mul_mi(cx<R> a) { return cx<R>{a.y, -a.x}; }     // a * (-i)
// a * i * sign (sign = +1 or -1 at compile time)
template <int SIGN, class R> WF_D cx<R> mul_si(cx<R> a) {
  return SIGN > 0 ? mul_i(a) : mul_mi(a);
}

// loads/stores between FP64 / FP32 storage and the arithmetic type
template <class R> WF_D cx<R> ld_c(const double2* p) {
  double2 v = *p;
  return cx<R>{RT<R>::from_d(v.x), RT<R>::from_d(v.y)};
}
template <class R> WF_D cx<R> ld_c(const float2* p) {
  float2 v = *p;
  return cx<R>{RT<R>::from_f(v.x), RT<R>::from_f(v.y)};
}
template <class R> WF_D void st_c(double2* p, cx<R> v) { *p = make_double2(RT<R>::to_d(v.x), RT<R>::to_d(v.y)); }
template <class R> WF_D void st_c(float2* p, cx<R> v) { *p = make_float2(RT<R>::to_f(v.x), RT<R>::to_f(v.y)); }

// storage complex type for an arithmetic type
template <class R> struct Store { using T = double2; using S = double; };
template <> struct Store<float> { using T = float2; using S = float; };

// ------------------------------------------------------------------------------------------
// dot-product accumulation.  For FP32 data the products are formed exactly (two-product) and
// accumulated in double-float; for FP64 data in FP64.  Either way the per-thread partial is
// returned as a double and the cross-thread sums are FP64.  Sums whose terms are all >= 0 (norms,
// <p, m p>, sum D T^2) add a 16-byte vector's few terms in the storage type first and pass that
// partial to add(): no cancellation, so the relative error stays a few units of FP32 rounding.
// ------------------------------------------------------------------------------------------
struct AccD {
  double s = 0.0;
  WF_D void add_prod(double a, double b) { s = fma(a, b, s); }
  WF_D void add(double a) { s += a; }
  WF_D double get() const { return s; }
};
struct AccF {
  float hi = 0.f, lo = 0.f;
  WF_D void add_prod(float a, float b) {
    float p = __fmul_rn(a, b);
    float e = __fmaf_rn(a, b, -p);
    float s, t;
    two_sum(hi, p, s, t);
    lo = __fadd_rn(lo, __fadd_rn(t, e));
    hi = s;
  }
  WF_D void add(float a) {
    float s, t;
    two_sum(hi, a, s, t);
    lo = __fadd_rn(lo, t);
    hi = s;
  }
  WF_D double get() const { return (double)hi + (double)lo; }
};
template <class S> struct AccFor { using T = AccD; };
template <> struct AccFor<float> { using T = AccF; };

// the lanes of this thread's warp that exist (a CTA's last warp may be partial)
WF_D int warp_lanes() {
  const int left = (int)blockDim.x - (int)(threadIdx.x & ~31u);
  return left < 32 ? left : 32;
}
WF_D unsigned lane_mask(int lanes) { return lanes == 32 ? 0xffffffffu : (1u << lanes) - 1u; }

// Block-wide sum of a double; result valid in thread 0.  `red` holds >= 32 doubles.
WF_D double block_sum(double v, double* red) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nl = warp_lanes();
  const unsigned mask = lane_mask(nl);
  for (int o = 16; o > 0; o >>= 1) {
    const double t = __shfl_down_sync(mask, v, o);
    if (l + o < nl) v += t;
  }
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  v = (threadIdx.x < nw) ? red[threadIdx.x] : 0.0;
  if (w == 0)
    for (int o = 16; o > 0; o >>= 1) {
      const double t = __shfl_down_sync(mask, v, o);
      if (l + o < nl) v += t;
    }
  return v;
}

// ------------------------------------------------------------------------------------------
// Chained launches.  A kernel launched with programmatic stream serialisation (Ctx::chain) starts as soon as the
// last CTA of its predecessor is done, before that one's memory is flushed and its completion signalled;
// chain_start() waits for the latter.  Only constants (twiddles, tensor maps) may be touched before it.  Launched
// plainly it does nothing.  (Letting the successor start earlier still, griddepcontrol.launch_dependents at the
// start of each kernel, is slower: its waiting CTAs crowd the SMs that drain first.  Mixed solve at 64^3: 4.54 ms
// plain, 4.33 here, 4.72 with early starts; at 512^3 290, 290, 328.)
// ------------------------------------------------------------------------------------------
WF_D void chain_start() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The last CTA of a grid (of `total` CTAs that all call this, after thread 0 has written the CTA's partial
// sums) gets true, with every other CTA's partial sums visible; *ticket is 0 before and after.
WF_D bool last_cta(unsigned* ticket, unsigned total) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(ticket, 1u) == total - 1;
    if (last) {
      *ticket = 0;
      __threadfence();
    }
  }
  __syncthreads();
  return last;
}
