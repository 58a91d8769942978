// Amplitude stage of the tensor-core path, phased (layout: phased.h): a CTA
// per event, every stored wavefunction once per helicity pattern of its legs
// in shared memory, every diagram amplitude written out for the
// colour-amplitude GEMM (jamp_gemm.cu) with the row maxima and the
// cancellation mass.
//
// What bounds it: the issue slots of the FP32 contractions.  gg>5g has 7245 x
// 112 diagram amplitudes per event, 30 instructions each (a complex dot of
// four components, its sign, maxima, mass and store), and 3060 x 32 currents
// of five legs at about 110, together some 1.3 M warp instructions per event.
// An interpreter lane pays for every operation its own decoding, its own
// index arithmetic and the latency of its own input loads on top; here a unit
// fixes operation, leg sets and lane-to-variant maps once for its whole list,
// OUTER units hold four partials in registers while the free wavefunctions
// stream by (16 bytes of shared memory per contraction and lane instead of
// 64), and FUSED units evaluate a five-leg current once for its 32 helicity
// patterns instead of once for each of the 112 combinations and never store
// it.  Measured on GB300 in microseconds per event (best per-lane,
// helicity-shared or split shape before, this kernel): gg>5g 9.09, 3.13;
// uu~>5g 1.50, 0.70; uu>uu+3g 0.52, 0.33; gg>4g 0.28, 0.16; uu~>4g 0.056,
// 0.051.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "../../include/mea.h"
#include "amp_common.cuh"
#include "heget.cuh"
#include "kernels.h"
#include "phased.h"

namespace mea {
namespace {

union PhUnitWords {
  uint4 v;
  PhUnit u;
};
union PhItemWords {
  uint4 v;
  PhItem r;
};
union PhHeadWords {
  uint4 v;
  PhOuterHead r;
};
union PhOuterWords {
  uint4 v[2];
  PhOuterRec r;
};
union PhFusedWords {
  uint4 v[2];
  PhFusedRec r;
};
union PhGenericWords {
  uint4 v[2];
  PhGenericRec r;
};

__device__ __forceinline__ W4<float> ph_ld(const float* area, uint32_t idx) {
  const float4 u = *reinterpret_cast<const float4*>(area + idx * 8);
  const float4 v = *reinterpret_cast<const float4*>(area + idx * 8 + 4);
  W4<float> w;
  w.c[0] = {u.x, u.y}; w.c[1] = {u.z, u.w}; w.c[2] = {v.x, v.y}; w.c[3] = {v.z, v.w};
  return w;
}
__device__ __forceinline__ void ph_st(float* area, uint32_t idx, const W4<float>& w) {
  *reinterpret_cast<float4*>(area + idx * 8) = make_float4(w.c[0].r, w.c[0].i, w.c[1].r, w.c[1].i);
  *reinterpret_cast<float4*>(area + idx * 8 + 4) = make_float4(w.c[2].r, w.c[2].i, w.c[3].r, w.c[3].i);
}

// maximum that keeps a NaN (a non-finite amplitude marks its row)
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// What a unit needs of its event.
struct PhEvent {
  float* area;       // variants
  const float* et;   // leg blocks of the event table
  const float* mt;   // mask rows
  char* out;         // amplitude (Re, Im) of combination 0, diagram 0
  uint32_t lda4;     // bytes between diagrams
  int* mx_re;        // [H] row maxima as integers
  int* mx_im;
  float* mass;       // [H] this unit's accumulator
  float g, gg;
};

// One lane's running maxima and mass over a unit's amplitudes of one combination.
struct PhAcc {
  float re = 0.f, im = 0.f, mass = 0.f;
  // amplitude a of diagram d (bit 15: negated) with weight w, to out + 8 h
  __device__ __forceinline__ void take(cx<float> a, uint32_t d, float w, char* out_h, uint32_t lda4) {
    const uint32_t sg = (d & 0x8000u) << 16;
    a.r = __uint_as_float(__float_as_uint(a.r) ^ sg);
    a.i = __uint_as_float(__float_as_uint(a.i) ^ sg);
    *reinterpret_cast<float2*>(out_h + (size_t)(d & 0x7fffu) * lda4) = make_float2(a.r, a.i);
    const float ar = fabsf(a.r), ai = fabsf(a.i);
    re = max_nan(re, ar);
    im = max_nan(im, ai);
    mass += w * (ar + ai);
  }
  __device__ __forceinline__ void flush(const PhEvent& E, int h) const {
    atomicMax(E.mx_re + h, __float_as_int(re));  // non-negative floats (and NaN) order as integers
    atomicMax(E.mx_im + h, __float_as_int(im));
    E.mass[h] += mass;
  }
};

template <int OP>
__device__ __forceinline__ W4<float> ph_current(const W4<float>& a, const W4<float>& b, const W4<float>& c, const float* mt,
                                                const uint8_t* r, const PhEvent& E) {
  const float* q = mt + 5 * r[2];
  if constexpr (OP == OP_JVV) return jvv<float>(a, b, mt + 5 * r[0], mt + 5 * r[1], q[4], E.g);
  else if constexpr (OP == OP_JGGG) return jggg<float>(a, b, c, q[4], E.gg);
  else if constexpr (OP == OP_FVI) return fvi<float>(a, b, q, q[4], E.g);
  else if constexpr (OP == OP_FVO) return fvo<float>(a, b, q, q[4], E.g);
  else return jio<float>(a, b, q[4], E.g);
}

template <int OP>
__device__ __forceinline__ void ph_produce(const PhUnit& u, const uint4* rec, const DevProgram& P, const PhEvent& E,
                                           int lane) {
  for (int i = lane; i < u.n; i += 32) {
    PhItemWords it;
    it.v = __ldg(rec + i);
    const PhItem& r = it.r;
    W4<float> x;
    if constexpr (OP == OP_EXT) {
      const int l = r.x & 15;
      const int type = P.leg_info[4 * l], kind = P.leg_info[4 * l + 1];
      const bool in = P.leg_info[4 * l + 2] != 0;
      const float* o = E.et + 8 * l;
      const int h = (r.x >> 4) ? 1 : -1;
      if (type == 0) x = ext_gluon<float>(o, o + 3, h, !in);
      else x = ext_spinor<float>(o[0], o[1], mk<float>(o[2], o[3]), h, kind);
    } else {
      const W4<float> a = ph_ld(E.area, r.in[0]), b = ph_ld(E.area, r.in[1]);
      if constexpr (OP == OP_JGGG) {
        x = ph_current<OP>(a, b, ph_ld(E.area, r.in[2]), E.mt, r.r, E);
      } else if constexpr (OP == OP_PVVV) {
        x = vvv_part<float>(a, b, E.mt + 5 * r.r[0], E.mt + 5 * r.r[1], E.mt + 5 * r.r[2], E.g);
      } else if constexpr (OP == OP_PGGGG) {
        x = gggg_part<float>(a, b, ph_ld(E.area, r.in[2]), E.gg);
      } else if constexpr (OP == OP_PIOV) {
        x = r.x == 0 ? iov_part_i<float>(a, b, E.g) : (r.x == 1 ? iov_part_o<float>(a, b, E.g) : iov_part_v<float>(a, b, E.g));
      } else {
        x = ph_current<OP>(a, b, a, E.mt, r.r, E);
      }
    }
    ph_st(E.area, r.out, x);
  }
}

template <bool PLAIN>
__device__ __forceinline__ void ph_outer(const PhUnit& u, const uint4* rec, const uint8_t* hv, int H, const PhEvent& E,
                                         int lane) {
  const int h = 32 * u.pass + lane;
  const bool on = h < H;
  const int hc = on ? h : 0;
  const uint32_t vf = __ldg(hv + 128 * u.sf + hc), vp = __ldg(hv + 128 * u.sp + hc);
  PhHeadWords hd;
  hd.v = __ldg(rec);
  W4<float> p[kPhPartials];
#pragma unroll
  for (int k = 0; k < kPhPartials; ++k) p[k] = ph_ld(E.area, hd.r.p[k < u.np ? k : 0] + vp);
  char* out = E.out + 8 * hc;
  PhAcc acc;
  PhOuterWords nx;
  nx.v[0] = __ldg(rec + 1);
  nx.v[1] = __ldg(rec + 2);
  for (int i = 0; i < u.n; ++i) {
    const PhOuterWords c = nx;
    if (i + 1 < u.n) {
      nx.v[0] = __ldg(rec + 2 * i + 3);
      nx.v[1] = __ldg(rec + 2 * i + 4);
    }
    const W4<float> w = ph_ld(E.area, c.r.f + vf);
#pragma unroll
    for (int k = 0; k < kPhPartials; ++k)
      if (k < u.np) {
        const cx<float> a = part_contract<float>(w, p[k], PLAIN, false);
        if (on) acc.take(a, c.r.d[k], c.r.w[k], out, E.lda4);
      }
  }
  if (on) acc.flush(E, h);
}

template <int OP>
__device__ __forceinline__ void ph_fused(const PhUnit& u, const uint4* rec, const PhSet* set, const PhEvent& E, int lane) {
  const int lg = u.lanes, per = 32 >> lg, slot = lane >> lg;
  const uint8_t* sub = &set->sub[0][0] + lane;
  uint32_t uo[kPhRounds], hh[kPhRounds];
#pragma unroll
  for (int r = 0; r < kPhRounds; ++r) {
    const uint32_t x = __ldg(&set->uh[r][lane]);
    uo[r] = x & 0xffu;
    hh[r] = x == kPhNone ? 0xffffu : x >> 8;
  }
  PhAcc acc[kPhRounds];
  for (int t = slot; t < u.n; t += per) {
    PhFusedWords c;
    c.v[0] = __ldg(rec + 2 * t);
    c.v[1] = __ldg(rec + 2 * t + 1);
    const W4<float> a = ph_ld(E.area, c.r.in[0] + __ldg(sub + 32 * c.r.m[0]));
    const W4<float> b = ph_ld(E.area, c.r.in[1] + __ldg(sub + 32 * c.r.m[1]));
    W4<float> x;
    if constexpr (OP == OP_JGGG) x = ph_current<OP>(a, b, ph_ld(E.area, c.r.in[2] + __ldg(sub + 32 * c.r.m[2])), E.mt, c.r.r, E);
    else x = ph_current<OP>(a, b, a, E.mt, c.r.r, E);
#pragma unroll
    for (int r = 0; r < kPhRounds; ++r)
      if (hh[r] != 0xffffu) {
        const W4<float> p = ph_ld(E.area, c.r.p + uo[r]);
        const cx<float> s = part_contract<float>(x, p, c.r.plain != 0, false);
        acc[r].take(s, c.r.d, c.r.w, E.out + 8 * hh[r], E.lda4);
      }
  }
  // the slots of a warp share combinations: one slot at a time (max and sum in slot order)
  for (int s = 0; s < per; ++s) {
    if (slot == s)
#pragma unroll
      for (int r = 0; r < kPhRounds; ++r)
        if (hh[r] != 0xffffu) acc[r].flush(E, (int)hh[r]);
    __syncwarp();
  }
}

__device__ __forceinline__ void ph_generic(const PhUnit& u, const uint4* rec, const uint8_t* hv, int H, const PhEvent& E,
                                           int lane) {
  const int h = 32 * u.pass + lane;
  if (h < H) {
    PhAcc acc;
    for (int i = 0; i < u.n; ++i) {
      PhGenericWords c;
      c.v[0] = __ldg(rec + 2 * i);
      c.v[1] = __ldg(rec + 2 * i + 1);
      auto in = [&](int k) { return ph_ld(E.area, c.r.in[k] + __ldg(hv + 128 * c.r.m[k] + h)); };
      cx<float> s;
      switch (c.r.type) {
        case OP_AVVV: {
          const W4<float> a = in(0), b = in(1), d = in(2);
          s = vvv_amp<float>(a, b, d, E.mt + 5 * c.r.r[0], E.mt + 5 * c.r.r[1], E.mt + 5 * c.r.r[2], E.g);
          break;
        }
        case OP_AGGGG: {
          const W4<float> a = in(0), b = in(1), d = in(2), e = in(3);
          s = gggg_amp<float>(a, b, d, e, E.gg);
          break;
        }
        case OP_AIOV: {
          const W4<float> a = in(0), b = in(1), d = in(2);
          s = iov_amp<float>(a, b, d, E.g);
          break;
        }
        default: {
          const W4<float> a = in(0), b = in(1);
          s = part_contract<float>(a, b, (c.r.flags & 1u) != 0, (c.r.flags & 2u) != 0);
          break;
        }
      }
      acc.take(s, c.r.d, c.r.w, E.out + 8 * h, E.lda4);
    }
    acc.flush(E, h);
  }
}

// Shared memory of a CTA: the area, the event table, row maxima [2][H], the
// mass accumulators [kPhMassSlots][H], input-check bits.
__host__ __device__ __forceinline__ size_t ph_smem(int area, int tab, int H) {
  size_t b = (size_t)area * 32;
  b += ((size_t)tab * 4 + 15) & ~size_t(15);
  b += (size_t)(2 + kPhMassSlots) * H * 4;
  return b + 16;
}

// Unit i of the program always adds into mass accumulator i mod kPhMassSlots,
// and the number of warps divides kPhMassSlots, so an accumulator belongs to
// one warp, takes its units in the same order for every CTA size, and the
// result does not depend on the launch shape.
__global__ void __launch_bounds__(32 * kPhMassSlots, 1) amp_phased_kernel(const DevProgram P, const AmpLaunch A,
                                                                          const AmpConfig C) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int t = threadIdx.x, lane = t & 31, W = blockDim.x >> 5, H = C.H, n_ext = P.n_ext;
  const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);
  const int tab_stride = event_table_stride(n_ext, P.n_masks);
  float* tab = reinterpret_cast<float*>(smem + (size_t)P.ph_area * 32);
  int* mx = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(tab) + (((size_t)tab_stride * 4 + 15) & ~size_t(15)));
  float* mass = reinterpret_cast<float*>(mx + 2 * H);
  unsigned int* evflag = reinterpret_cast<unsigned int*>(mass + kPhMassSlots * H);
  PhEvent E;
  E.area = reinterpret_cast<float*>(smem);
  E.et = tab;
  E.mt = tab + 8 * n_ext;
  E.lda4 = (uint32_t)(A.lda * 4);
  E.mx_re = mx;
  E.mx_im = mx + H;
  E.g = (float)P.g;
  E.gg = (float)(P.g * P.g);
  const uint4* units = reinterpret_cast<const uint4*>(P.ph_units);
  const uint4* rec = reinterpret_cast<const uint4*>(P.ph_rec);

  for (int64_t ev = blockIdx.x; ev < A.n_events; ev += gridDim.x) {
    if (t == 0) *evflag = 0u;
    for (int i = t; i < (2 + kPhMassSlots) * H; i += blockDim.x) mx[i] = 0;
    __syncthreads();
    tile_prep<float>(P, A, tab, tab_stride, ev, A.n_events, 1, t, blockDim.x, evflag);
    __syncthreads();
    E.out = reinterpret_cast<char*>(A.amp_out + 2 * ev * H);
    int u0 = 0;
    for (int ph = 0; ph < P.ph_phases; ++ph) {
      const int u1 = __ldg(P.ph_end + ph);
      // the warp's first unit of this phase: index = warp (mod W)
      int i = u0 + (warp - u0 % W + W) % W;
      for (; i < u1; i += W) {
        PhUnitWords c;
        c.v = __ldg(units + i);
        const uint4* r = rec + c.u.rec;
        E.mass = mass + (i % kPhMassSlots) * H;
        if (c.u.type == PH_OUTER) {
          if (c.u.op) ph_outer<true>(c.u, r, P.ph_hv, H, E, lane);
          else ph_outer<false>(c.u, r, P.ph_hv, H, E, lane);
        } else if (c.u.type == PH_FUSED) {
          const PhSet* s = P.ph_sets + c.u.set;
          switch (c.u.op) {
            case OP_JVV: ph_fused<OP_JVV>(c.u, r, s, E, lane); break;
            case OP_JGGG: ph_fused<OP_JGGG>(c.u, r, s, E, lane); break;
            case OP_FVI: ph_fused<OP_FVI>(c.u, r, s, E, lane); break;
            case OP_FVO: ph_fused<OP_FVO>(c.u, r, s, E, lane); break;
            default: ph_fused<OP_JIO>(c.u, r, s, E, lane); break;
          }
        } else if (c.u.type == PH_PRODUCE) {
          switch (c.u.op) {
            case OP_EXT: ph_produce<OP_EXT>(c.u, r, P, E, lane); break;
            case OP_JVV: ph_produce<OP_JVV>(c.u, r, P, E, lane); break;
            case OP_JGGG: ph_produce<OP_JGGG>(c.u, r, P, E, lane); break;
            case OP_FVI: ph_produce<OP_FVI>(c.u, r, P, E, lane); break;
            case OP_FVO: ph_produce<OP_FVO>(c.u, r, P, E, lane); break;
            case OP_JIO: ph_produce<OP_JIO>(c.u, r, P, E, lane); break;
            case OP_PVVV: ph_produce<OP_PVVV>(c.u, r, P, E, lane); break;
            case OP_PGGGG: ph_produce<OP_PGGGG>(c.u, r, P, E, lane); break;
            default: ph_produce<OP_PIOV>(c.u, r, P, E, lane); break;
          }
        } else {
          ph_generic(c.u, r, P.ph_hv, H, E, lane);
        }
        __syncwarp();  // the unit's mass is in its accumulator before the next unit adds
      }
      u0 = u1;
      __syncthreads();
    }
    for (int h = t; h < H; h += blockDim.x) {
      float m = 0.f;
      for (int k = 0; k < kPhMassSlots; ++k) m += mass[k * H + h];
      const float re = __int_as_float(E.mx_re[h]), im = __int_as_float(E.mx_im[h]);
      const bool fin = isfinite(re) && isfinite(im);
      const float nan = __int_as_float(0x7fc00000);
      const int64_t pair = ev * H + h;
      *reinterpret_cast<float2*>(A.amp_rowmax + 2 * pair) = make_float2(fin ? re : nan, fin ? im : nan);
      A.pair_kappa[pair] = m;  // divided by sum |J| after the colour-amplitude stage
    }
    if (t == 0) A.ev_flags[ev] = (uint8_t)*evflag;
    __syncthreads();  // the table and the accumulators are read until here
  }
}

}  // namespace

bool phased_supported(const DevProgram& p, bool fp64, int H) {
  return !fp64 && p.ph_units != nullptr && p.n_colour == 0 && H == p.ph_H;
}

int phased_max_area(const Program& P, int H, size_t max_smem) {
  const size_t rest = ph_smem(0, event_table_stride(P.n_ext, (int)P.masks.size()), H);
  return rest < max_smem ? (int)((max_smem - rest) / 32) : 0;
}

std::vector<AmpConfig> phased_candidates(const DevProgram& p, int H, int64_t n_events, int num_sms, size_t max_smem,
                                         size_t smem_per_sm) {
  std::vector<AmpConfig> out;
  const size_t sm = ph_smem(p.ph_area, event_table_stride(p.n_ext, p.n_masks), H);
  cudaFuncAttributes fa;
  if (sm > max_smem || cudaFuncGetAttributes(&fa, (const void*)amp_phased_kernel) != cudaSuccess) {
    cudaGetLastError();
    return out;
  }
  const int regs_warp = ((std::max(fa.numRegs, 1) + 7) / 8) * 8 * 32;
  for (int W : {2, 3, 4, 6, 8, 12, 24}) {
    const int res = std::min({65536 / (regs_warp * W), (int)(smem_per_sm / (sm + 1024)), 64 / W, 32});
    if (res < 1) continue;
    AmpConfig c;
    c.H = H;
    c.E_cta = 1;
    c.threads = 32 * W;
    c.smem = sm;
    c.phased = true;
    c.per_sm = res;
    c.grid = (int)std::min<int64_t>((int64_t)res * num_sms, std::max<int64_t>(n_events, 1));
    out.push_back(c);
  }
  return out;
}

const AmpConfig* phased_default(const std::vector<AmpConfig>& cands) {
  const AmpConfig* best = &cands.front();  // the most resident warps
  for (const AmpConfig& c : cands)
    if (c.per_sm * c.threads > best->per_sm * best->threads) best = &c;
  return best;
}

cudaError_t launch_amp_phased(const DevProgram& p, const AmpConfig& c, const AmpLaunch& a, cudaStream_t s) {
  const int W = c.threads / 32;
  if (!phased_supported(p, false, c.H) || !a.amp_out || a.event_list || a.hel_mode != 0) return cudaErrorInvalidValue;
  // 32-bit byte strides between diagrams; float2 stores of the row maxima
  if (a.lda > kPhasedMaxLda || c.E_cta != 1 || c.threads % 32 != 0 || W < 1 || W > kPhMassSlots || kPhMassSlots % W != 0 ||
      c.smem != ph_smem(p.ph_area, event_table_stride(p.n_ext, p.n_masks), c.H))
    return cudaErrorInvalidConfiguration;
  cudaError_t e = ensure_dynamic_smem((const void*)amp_phased_kernel, c.smem);
  if (e != cudaSuccess) return e;
  if (cudaFuncSetAttribute(amp_phased_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, carveout_percent(c)) !=
      cudaSuccess)
    cudaGetLastError();
  amp_phased_kernel<<<c.grid, c.threads, c.smem, s>>>(p, a, c);
  return cudaGetLastError();
}

}  // namespace mea
