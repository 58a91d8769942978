// Amplitude stage of the tensor-core path, phased (layout: phased.h): a CTA
// per event, every stored wavefunction once per helicity pattern of its legs
// in shared memory, every diagram amplitude written out for the
// colour-amplitude GEMM (jamp_gemm.cu) with the row maxima and the
// cancellation mass.
//
// What bounds it: the issue slots of the FP32 contractions, and behind them
// instruction fetch.  gg>5g has 7245 x 112 diagram amplitudes per event, a
// complex dot of four components with its maxima, mass and store each, and
// 3060 x 32 currents of five legs at about 110 instructions.  An interpreter
// lane pays for every operation its own decoding, its own index arithmetic and
// the latency of its own input loads on top; here a unit fixes operation, leg
// sets and lane-to-variant maps once for its whole list, OUTER units hold four
// partials in registers while the free wavefunctions stream by (16 bytes of
// shared memory per contraction and lane instead of 64), and FUSED units
// evaluate a five-leg current once for its 32 helicity patterns instead of
// once for each of the 112 combinations and never store it.  Records hold byte
// offsets that are added as they are, the vertex functions are written out
// (vertex_pinned.cuh) so that momenta come in 16-byte loads, 80 registers leave
// two CTAs of 12 warps on an SM without spills, a phase's units are dealt to
// the warps by cost, and a FUSED unit stops after its last round.  Code that
// is added costs: a second instantiation of the gluon currents without the
// test per round took gg>5g from 1.33 to 1.81 (the code no longer fits the
// instruction caches), unrolling OUTER by two gg>4g from 0.067 to 0.071.
// Measured on GB300 in microseconds per event (best per-lane, helicity-shared
// or split shape; a warp list without those measures; this kernel): gg>5g 4.6,
// 1.87, 1.32; uu~>5g 1.50, 0.70, 0.59; uu>uu+3g 0.52, 0.34, 0.25; gg>4g 0.15,
// 0.106, 0.067; uu~>4g 0.056, 0.051, 0.033.  (The pure gluons with every
// helicity combination of a flipped pair: twice that.)
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "../../include/mea.h"
#include "amp_common.cuh"
#include "heget.cuh"
#include "kernels.h"
#include "phased.h"
#include "vertex_pinned.cuh"

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
union PhOuterWords {
  uint4 v[3];
  PhOuterRec r;
};
union PhFusedWords {
  uint4 v[3];
  PhFusedRec r;
};
union PhGenericWords {
  uint4 v[2];
  PhGenericRec r;
};

__device__ __forceinline__ W4<float> ph_at(const unsigned char* p) {
  const float4 u = *reinterpret_cast<const float4*>(p);
  const float4 v = *reinterpret_cast<const float4*>(p + 16);
  W4<float> w;
  w.c[0] = {u.x, u.y}; w.c[1] = {u.z, u.w}; w.c[2] = {v.x, v.y}; w.c[3] = {v.z, v.w};
  return w;
}
__device__ __forceinline__ void ph_st(unsigned char* p, const W4<float>& w) {
  *reinterpret_cast<float4*>(p) = make_float4(w.c[0].r, w.c[0].i, w.c[1].r, w.c[1].i);
  *reinterpret_cast<float4*>(p + 16) = make_float4(w.c[2].r, w.c[2].i, w.c[3].r, w.c[3].i);
}
// a row of the event table: momentum and 1/P^2
struct PhRow {
  float k[4];
  __device__ __forceinline__ explicit PhRow(const unsigned char* p) {
    const float4 u = *reinterpret_cast<const float4*>(p);
    k[0] = u.x; k[1] = u.y; k[2] = u.z; k[3] = u.w;
  }
};
__device__ __forceinline__ float ph_inv(const unsigned char* p) { return *reinterpret_cast<const float*>(p + 16); }

// What a unit needs of its event.
struct PhEvent {
  unsigned char* area;       // variants, 32 bytes each
  const unsigned char* mt;   // mask rows, 32 bytes each
  const float* et;           // leg blocks of the event table
  char* out;                 // amplitude (Re, Im) of combination 0, row 0
  uint32_t lda4;             // bytes between rows
  int* mx_re;                // [H] row maxima as integers
  int* mx_im;
  float* mass;               // [H] this unit's accumulator
  float g, gg;
};

// One lane's running maxima and mass over a unit's amplitudes of one
// combination.  A non-finite amplitude makes the mass non-finite.
struct PhAcc {
  float re = 0.f, im = 0.f, mass = 0.f;
  // amplitude a with weight w, stored at `to` where `on`
  __device__ __forceinline__ void take(cx<float> a, float w, char* to, bool on) {
    if (on) *reinterpret_cast<float2*>(to) = make_float2(a.r, a.i);
    re = fmaxf(re, fabsf(a.r));
    im = fmaxf(im, fabsf(a.i));
    mass += w * (fabsf(a.r) + fabsf(a.i));
  }
  __device__ __forceinline__ void flush(const PhEvent& E, int h) const {
    atomicMax(E.mx_re + h, __float_as_int(re));  // non-negative floats order as integers
    atomicMax(E.mx_im + h, __float_as_int(im));
    E.mass[h] += mass;
  }
};

// Current of one op type; r: byte offsets of its rows.
template <int OP>
__device__ __forceinline__ W4<float> ph_current(const W4<float>& a, const W4<float>& b, const W4<float>& c, uint32_t r0,
                                                uint32_t r1, uint32_t r2, const PhEvent& E) {
  const float inv = ph_inv(E.mt + r2);
  if constexpr (OP == OP_JVV) {
    const PhRow p(E.mt + r0), q(E.mt + r1);
    return pinned::jvv(a, b, p.k, q.k, inv, E.g);
  } else if constexpr (OP == OP_JGGG) {
    return pinned::jggg(a, b, c, inv, E.gg);
  } else if constexpr (OP == OP_FVI) {
    const PhRow q(E.mt + r2);
    return pinned::fvi(a, b, q.k, inv, E.g);
  } else if constexpr (OP == OP_FVO) {
    const PhRow q(E.mt + r2);
    return pinned::fvo(a, b, q.k, inv, E.g);
  } else {
    return pinned::jio(a, b, inv, E.g);
  }
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
      const W4<float> a = ph_at(E.area + 32u * r.in[0]), b = ph_at(E.area + 32u * r.in[1]);
      if constexpr (OP == OP_JGGG) {
        x = ph_current<OP>(a, b, ph_at(E.area + 32u * r.in[2]), 0, 0, 32u * r.r[2], E);
      } else if constexpr (OP == OP_PVVV) {
        const PhRow k0(E.mt + 32u * r.r[0]), k1(E.mt + 32u * r.r[1]), k2(E.mt + 32u * r.r[2]);
        x = pinned::vvv_part(a, b, k0.k, k1.k, k2.k, E.g);
      } else if constexpr (OP == OP_PGGGG) {
        x = pinned::gggg_part(a, b, ph_at(E.area + 32u * r.in[2]), E.gg);
      } else if constexpr (OP == OP_PIOV) {
        x = r.x == 0 ? pinned::iov_part_i(a, b, E.g) : (r.x == 1 ? pinned::iov_part_o(a, b, E.g) : pinned::iov_part_v(a, b, E.g));
      } else {
        x = ph_current<OP>(a, b, a, 32u * r.r[0], 32u * r.r[1], 32u * r.r[2], E);
      }
    }
    ph_st(E.area + 32u * r.out, x);
  }
}

template <bool PLAIN, int NP>
__device__ __forceinline__ void ph_outer(const PhUnit& u, const uint4* rec, const uint8_t* hv, int H, const PhEvent& E,
                                         int lane) {
  const int h = 32 * u.pass + lane;
  const bool on = h < H;
  const int hc = on ? h : 0;
  const unsigned char* wf = E.area + 32u * __ldg(hv + 128 * u.sf + hc);
  const unsigned char* wp = E.area + 32u * __ldg(hv + 128 * u.sp + hc);
  const uint4 hd = __ldg(rec);
  const uint32_t hp[4] = {hd.x, hd.y, hd.z, hd.w};
  W4<float> p[NP];
#pragma unroll
  for (int k = 0; k < NP; ++k) p[k] = ph_at(wp + hp[k]);
  char* out = E.out + 8 * hc;
  PhAcc acc;
#pragma unroll 1
  for (int i = 0; i < u.n; ++i) {
    PhOuterWords c;
#pragma unroll
    for (int k = 0; k < 3; ++k) c.v[k] = __ldg(rec + 3 * i + 1 + k);
    const W4<float> w = ph_at(wf + c.r.f);
#pragma unroll
    for (int k = 0; k < NP; ++k) acc.take(pinned::dot<PLAIN>(w, p[k]), c.r.w[k], out + (size_t)c.r.d[k] * E.lda4, on);
  }
  if (on) acc.flush(E, h);
}
template <bool PLAIN>
__device__ __forceinline__ void ph_outer_any(const PhUnit& u, const uint4* rec, const uint8_t* hv, int H, const PhEvent& E,
                                             int lane) {
  switch (u.np) {
    case 1: ph_outer<PLAIN, 1>(u, rec, hv, H, E, lane); break;
    case 2: ph_outer<PLAIN, 2>(u, rec, hv, H, E, lane); break;
    case 3: ph_outer<PLAIN, 3>(u, rec, hv, H, E, lane); break;
    default: ph_outer<PLAIN, 4>(u, rec, hv, H, E, lane); break;
  }
}

template <int OP>
__device__ __forceinline__ void ph_fused(const PhUnit& u, const uint4* rec, const PhSet* set, const PhEvent& E, int lane) {
  // a quark current closes with a spinor partial, a gluon current with a vector
  constexpr bool plain = OP == OP_FVI || OP == OP_FVO;
  const int lg = u.lanes, per = 32 >> lg, slot = lane >> lg;
  const char* sub = reinterpret_cast<const char*>(&set->sub[0][0] + lane);
  auto in = [&](uint32_t base, uint32_t m) {
    return ph_at(E.area + base + __ldg(reinterpret_cast<const uint16_t*>(sub + m)));
  };
  uint32_t uh[kPhRounds];  // partial's variant, combination << 8
#pragma unroll
  for (int r = 0; r < kPhRounds; ++r) uh[r] = __ldg(&set->uh[r][lane]);
  PhAcc acc[kPhRounds];
  for (int t = slot; t < u.n; t += per) {
    PhFusedWords c;
#pragma unroll
    for (int k = 0; k < 3; ++k) c.v[k] = __ldg(rec + 3 * t + k);
    const W4<float> a = in(c.r.in[0], c.r.m[0]), b = in(c.r.in[1], c.r.m[1]);
    W4<float> x;
    if constexpr (OP == OP_JGGG) x = ph_current<OP>(a, b, in(c.r.in[2], c.r.m[2]), 0, 0, c.r.r[2], E);
    else x = ph_current<OP>(a, b, a, c.r.r[0], c.r.r[1], c.r.r[2], E);
    char* row = E.out + (size_t)c.r.d * E.lda4;
    const unsigned char* p = E.area + c.r.p;
#pragma unroll
    for (int r = 0; r < kPhRounds; ++r) {
      if (r >= u.rounds) break;
      const bool on = uh[r] != kPhNoPair;
      const cx<float> s = pinned::dot<plain>(x, ph_at(p + (on ? 32u * (uh[r] & 0xffu) : 0u)));
      acc[r].take(s, c.r.w, row + 8 * (uh[r] >> 8), on);
    }
  }
  // the slots of a warp share combinations: one slot at a time (max and sum in slot order)
  for (int s = 0; s < per; ++s) {
    if (slot == s)
#pragma unroll
      for (int r = 0; r < kPhRounds; ++r)
        if (uh[r] != kPhNoPair) acc[r].flush(E, (int)(uh[r] >> 8));
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
      auto in = [&](int k) { return ph_at(E.area + 32u * (c.r.in[k] + __ldg(hv + 128 * c.r.m[k] + h))); };
      cx<float> s;
      switch (c.r.type) {
        case OP_AVVV: {
          const W4<float> a = in(0), b = in(1), d = in(2);
          const PhRow k0(E.mt + 32u * c.r.r[0]), k1(E.mt + 32u * c.r.r[1]), k2(E.mt + 32u * c.r.r[2]);
          s = pinned::vvv_amp(a, b, d, k0.k, k1.k, k2.k, E.g);
          break;
        }
        case OP_AGGGG: {
          const W4<float> a = in(0), b = in(1), d = in(2), e = in(3);
          s = pinned::gggg_amp(a, b, d, e, E.gg);
          break;
        }
        case OP_AIOV: {
          const W4<float> a = in(0), b = in(1), d = in(2);
          s = pinned::iov_amp(a, b, d, E.g);
          break;
        }
        default: {
          const W4<float> a = in(0), b = in(1);
          s = (c.r.flags & 1u) ? pinned::dot<true>(a, b) : pinned::dot<false>(a, b);
          break;
        }
      }
      acc.take(s, c.r.w, E.out + 8 * h + (size_t)c.r.d * E.lda4, true);
    }
    acc.flush(E, h);
  }
}

// Shared memory of a CTA: the area, the mask rows (momentum, 1/P^2, padded to
// 32 bytes for 16-byte loads), the event table, row maxima [2][H], the mass
// accumulators [kPhWarps][H], input-check bits.
__host__ __device__ __forceinline__ size_t ph_smem(int area, int n_masks, int tab, int H) {
  size_t b = (size_t)(area + n_masks) * 32;
  b += ((size_t)tab * 4 + 15) & ~size_t(15);
  b += (size_t)(2 + kPhWarps) * H * 4;
  return b + 16;
}

// The units of list l of every phase add into mass accumulator l, and the number
// of warps divides the number of lists, so an accumulator belongs to one warp,
// takes its units in the same order for every CTA size, and the result does not
// depend on the launch shape.
__global__ void __launch_bounds__(32 * kPhWarps, 2) amp_phased_kernel(const DevProgram P, const AmpLaunch A,
                                                                          const AmpConfig C) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int t = threadIdx.x, lane = t & 31, W = blockDim.x >> 5, H = C.H, n_ext = P.n_ext;
  const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);
  const int tab_stride = event_table_stride(n_ext, P.n_masks);
  unsigned char* rows = smem + (size_t)P.ph_area * 32;
  float* tab = reinterpret_cast<float*>(rows + (size_t)P.n_masks * 32);
  int* mx = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(tab) + (((size_t)tab_stride * 4 + 15) & ~size_t(15)));
  float* mass = reinterpret_cast<float*>(mx + 2 * H);
  unsigned int* evflag = reinterpret_cast<unsigned int*>(mass + kPhWarps * H);
  PhEvent E;
  E.area = smem;
  E.et = tab;
  E.mt = rows;
  E.lda4 = (uint32_t)(A.lda * 4);
  E.mx_re = mx;
  E.mx_im = mx + H;
  E.g = (float)P.g;
  E.gg = (float)(P.g * P.g);
  const uint4* units = reinterpret_cast<const uint4*>(P.ph_units);
  const uint4* rec = reinterpret_cast<const uint4*>(P.ph_rec);

  for (int64_t ev = blockIdx.x; ev < A.n_events; ev += gridDim.x) {
    if (t == 0) *evflag = 0u;
    for (int i = t; i < (2 + kPhWarps) * H; i += blockDim.x) mx[i] = 0;
    __syncthreads();
    tile_prep<float>(P, A, tab, tab_stride, ev, A.n_events, 1, t, blockDim.x, evflag);
    __syncthreads();
    for (int i = t; i < 5 * P.n_masks; i += blockDim.x)
      reinterpret_cast<float*>(rows)[8 * (i / 5) + i % 5] = tab[8 * n_ext + i];
    __syncthreads();
    E.out = reinterpret_cast<char*>(A.amp_out + 2 * ev * H);
    for (int ph = 0; ph < P.ph_phases; ++ph) {
      for (int l = warp; l < kPhWarps; l += W) {
      const int* end = P.ph_end + ph * kPhWarps + l;
      const int u1 = __ldg(end);
      E.mass = mass + l * H;
      for (int i = ph + l > 0 ? __ldg(end - 1) : 0; i < u1; ++i) {
        PhUnitWords c;
        c.v = __ldg(units + i);
        const uint4* r = rec + c.u.rec;
        if (c.u.type == PH_OUTER) {
          if (c.u.op) ph_outer_any<true>(c.u, r, P.ph_hv, H, E, lane);
          else ph_outer_any<false>(c.u, r, P.ph_hv, H, E, lane);
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
      }
      __syncthreads();
    }
    for (int h = t; h < H; h += blockDim.x) {
      float m = 0.f;
      for (int k = 0; k < kPhWarps; ++k) m += mass[k * H + h];
      const float re = __int_as_float(E.mx_re[h]), im = __int_as_float(E.mx_im[h]);
      const bool fin = isfinite(m);
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
  const size_t rest = ph_smem(0, (int)P.masks.size(), event_table_stride(P.n_ext, (int)P.masks.size()), H);
  return rest < max_smem ? (int)((max_smem - rest) / 32) : 0;
}

std::vector<AmpConfig> phased_candidates(const DevProgram& p, int H, int64_t n_events, int num_sms, size_t max_smem,
                                         size_t smem_per_sm) {
  std::vector<AmpConfig> out;
  const size_t sm = ph_smem(p.ph_area, p.n_masks, event_table_stride(p.n_ext, p.n_masks), H);
  cudaFuncAttributes fa;
  if (sm > max_smem || cudaFuncGetAttributes(&fa, (const void*)amp_phased_kernel) != cudaSuccess) {
    cudaGetLastError();
    return out;
  }
  const int regs_warp = ((std::max(fa.numRegs, 1) + 7) / 8) * 8 * 32;
  for (int W : {1, 2, 3, 4, 6, 12}) {
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
  if (a.lda > kPhasedMaxLda || c.E_cta != 1 || c.threads % 32 != 0 || W < 1 || W > kPhWarps || kPhWarps % W != 0 ||
      c.smem != ph_smem(p.ph_area, p.n_masks, event_table_stride(p.n_ext, p.n_masks), c.H))
    return cudaErrorInvalidConfiguration;
  cudaError_t e = ensure_dynamic_smem((const void*)amp_phased_kernel, c.smem);
  if (e != cudaSuccess) return e;
  if (cudaFuncSetAttribute(amp_phased_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, carveout_percent(p, c)) !=
      cudaSuccess)
    cudaGetLastError();
  amp_phased_kernel<<<c.grid, c.threads, c.smem, s>>>(p, a, c);
  return cudaGetLastError();
}

}  // namespace mea
