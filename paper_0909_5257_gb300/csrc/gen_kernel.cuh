// Kernel template for the straight-line per-process bodies that codegen.cpp
// emits.  Same tile structure as the interpreter (amp_kernel.cu): FP64
// preparation of the per-event tables in shared memory, one lane per
// (event, helicity) running the process body with all wavefunctions and
// colour amplitudes in registers, fixed-order helicity sum.  Only the
// per-event tables and the lane results use shared memory.
#pragma once
#include <type_traits>

#include "amp_common.cuh"

namespace mea {
namespace {

constexpr int kGenMaxThreads = 256;

// A colour amplitude under accumulation: FP64 plain, FP32 two-sum compensated
// (lo collects the rounding errors), PACKED with its real and imaginary parts as
// one pair, so that a compensated addition is 7 instructions instead of 14 (the
// same roundings).  The FP32 pipe and the spills of the long bodies bound these
// kernels: packed additions together with accumulating the base columns only take
// 2^20 events of gg>ggg from 6.77 to 4.22 ms (168 registers) and from 8.03 to
// 5.25 ms (128).  Which bodies are packed: codegen.cpp.
template <typename R, bool PACKED>
struct JSum {
  cx<R> hi{R(0), R(0)};
};
template <>
struct JSum<float, false> {
  cx<float> hi{0.f, 0.f}, lo{0.f, 0.f};
};
template <>
struct JSum<float, true> {
  unsigned long long hi = 0, lo = 0;
};

__device__ __forceinline__ unsigned long long jpack(cx<float> a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.r), "f"(a.i));
  return r;
}
__device__ __forceinline__ cx<float> junpack(unsigned long long v) {
  cx<float> a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.r), "=f"(a.i) : "l"(v));
  return a;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {  // a - b, rounded once
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(b), "l"(0xBF800000BF800000ull), "l"(a));
  return r;
}

// J += a
__device__ __forceinline__ void jadd(JSum<float, true>& J, unsigned long long a) {
  const unsigned long long s = add2(J.hi, a);
  const unsigned long long bp = sub2(s, J.hi);
  const unsigned long long e = add2(sub2(J.hi, sub2(s, bp)), sub2(a, bp));
  J.hi = s;
  J.lo = add2(J.lo, e);
}
__device__ __forceinline__ void jadd(JSum<float, true>& J, cx<float> a) { jadd(J, jpack(a)); }
__device__ __forceinline__ void jadd(JSum<float, false>& J, cx<float> a) {
  cx<float> s, e;
  two_sum(J.hi.r, a.r, s.r, e.r);
  two_sum(J.hi.i, a.i, s.i, e.i);
  J.hi = s;
  J.lo = J.lo + e;
}
template <bool PACKED>
__device__ __forceinline__ void jadd(JSum<double, PACKED>& J, cx<double> a) {
  J.hi.r += a.r;
  J.hi.i += a.i;
}
// J += x, J -= x for another compensated sum x
__device__ __forceinline__ void jadd(JSum<float, true>& J, const JSum<float, true>& x) {
  jadd(J, x.hi);
  J.lo = add2(J.lo, x.lo);
}
__device__ __forceinline__ void jsub(JSum<float, true>& J, const JSum<float, true>& x) {
  jadd(J, x.hi ^ 0x8000000080000000ull);
  J.lo = sub2(J.lo, x.lo);
}
__device__ __forceinline__ void jadd(JSum<float, false>& J, const JSum<float, false>& x) {
  jadd(J, x.hi);
  J.lo = J.lo + x.lo;
}
__device__ __forceinline__ void jsub(JSum<float, false>& J, const JSum<float, false>& x) {
  jadd(J, -x.hi);
  J.lo = J.lo - x.lo;
}

template <typename R>
__device__ __forceinline__ cx<R> neg(cx<R> a) {
  return cx<R>{-a.r, -a.i};
}

__device__ __forceinline__ cx<float> jfin(const JSum<float, true>& J) { return junpack(add2(J.hi, J.lo)); }
__device__ __forceinline__ cx<float> jfin(const JSum<float, false>& J) { return J.hi + J.lo; }
template <bool PACKED>
__device__ __forceinline__ cx<double> jfin(const JSum<double, PACKED>& J) { return J.hi; }

// Register-cap variants: MINB resident CTAs of MAXT threads per SM cap a
// thread at 65536 / (MAXT MINB) registers.  More registers spill less of the
// long straight-line body, fewer keep more warps resident, and which wins
// depends on the body, so the FP32 bodies come at 128 (256 threads, MINB 2),
// 85 (256, 3) and 168 (192, 2) registers and the autotuner picks.  Measured on
// 2^20 events, ms at 168 / 128 / 85: gg>ggg 4.22 / 5.25 / 6.95, gg>gg 0.91 /
// 0.76 / 0.66, uu~>gg 0.69 / 0.64 / 0.61.  The FP64 bodies come at 128.  A
// module that also held uncapped FP32 variants measured 25-45 % slower on the
// same 128-register kernel, so none is built.
template <typename R, typename Body, int MINB, int MAXT>
__global__ void __launch_bounds__(MAXT, MINB) gen_kernel(const DevProgram P, const AmpLaunch A,
                                                                   const AmpConfig C) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr bool F32 = std::is_same<R, float>::value;
  const int L = blockDim.x;
  const int t = threadIdx.x;
  const int n_ext = P.n_ext, H = C.H, E = C.E_cta;
  const int tab_stride = event_table_stride(n_ext, P.n_masks);
  R* tab = reinterpret_cast<R*>(smem);
  size_t off = ((size_t)E * tab_stride * sizeof(R) + 7) & ~size_t(7);
  double* res = reinterpret_cast<double*>(smem + off);
  off += (size_t)L * sizeof(double);
  float* kap = reinterpret_cast<float*>(smem + off);
  unsigned int* evflag = reinterpret_cast<unsigned int*>(kap + L);  // [E] input-check bits
  for (int i = t; i < E; i += L) evflag[i] = 0u;

  const bool listed = A.event_list != nullptr;
  const int64_t n = listed ? (int64_t)(*A.list_count) : A.n_events;
  const int64_t n_tiles = (n + E - 1) / E;
  const R g = (R)P.g;
  const R gg = (R)(P.g * P.g);

  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t ev0 = tile * E;
    __syncthreads();  // evflag cleared (first tile) / released by the previous finish
    tile_prep<R>(P, A, tab, tab_stride, ev0, n, E, t, L, evflag);
    __syncthreads();
    const int e = t / H, h = t - (t / H) * H;
    const int64_t ev = ev0 + e;
    const bool active = (t < E * H) && (ev < n);
    double val = 0.0;
    float kappa = 0.f;
    if (active) {
      const int64_t gev = listed ? (int64_t)A.event_list[ev] : ev;
      uint32_t lam = 0;
      for (int l = 0; l < n_ext; ++l) {
        int8_t v;
        if (A.hel_mode == 0) v = P.hel[h * n_ext + l];
        else if (A.hel_mode == 1) v = P.hel_all[h * n_ext + l];
        else v = A.hel_given[gev * n_ext + l];
        if (v > 0) lam |= 1u << l;
      }
      const R* et = tab + (size_t)e * tab_stride;
      Body::run(et, et + 8 * n_ext, lam, g, gg, P.cf_inv_den, val, kappa);
      if (!isfinite(val)) val = __longlong_as_double(0x7ff8000000000000ll);
    }
    res[t] = val;
    kap[t] = kappa;
    __syncthreads();
    tile_finish<F32>(A, t, E, H, ev0, n, listed, res, kap, evflag);
    __syncthreads();
  }
}

template <typename R, typename Body, int MINB, int MAXT>
void gen_launch_v(const DevProgram& p, const AmpConfig& plan, const AmpLaunch& a, cudaStream_t s) {
  auto k = gen_kernel<R, Body, MINB, MAXT>;
  // a listed launch's count is on the device: the plan's tiles
  const AmpConfig c = a.event_list ? plan : gen_spread(p, plan, a.n_events, sizeof(R));
  if (ensure_dynamic_smem((const void*)k, c.smem) != cudaSuccess) return;
  // the carveout is a preference: a value the driver refuses leaves the launch valid.  The
  // plan's, so that calls of several sizes do not reconfigure the SMs (uu~>ggg, 4096 events: 29 -> 37 us).
  if (cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, carveout_percent(p, plan)) != cudaSuccess)
    cudaGetLastError();
  k<<<c.grid, c.threads, c.smem, s>>>(p, a, c);
}

// Each kernel variant of a process -- the FP32 bodies (with vertex partials
// or one vertex call per diagram) at 128, 85 and 168 registers, numbered
// 2 * cap + body (kernels.h), and the FP64 body with partials at 128 -- is
// instantiated in a translation unit (device module) of its own by
// codegen.cpp, behind two plain functions: gen_launch_v and the kernel's
// address.  Separate units compile in parallel.
}  // namespace
}  // namespace mea
