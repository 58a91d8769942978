// FP64 path: |M|^2 by the ordered recursion (ordered.h, ordered_eval.cuh).
//
// A CTA owns a tile of E events.  Phase 0 is the other kernels' (tile_prep,
// amp_common.cuh).  Then the stages run one after another, the threads taking
// (event, word, helicity pattern) items in turn, with a CTA barrier where the
// level grows; then the colour sum, a thread per (event, combination, share of
// the matrix rows); then the helicity sum and the flags (tile_finish).
//
// Bound by the FP64 pipe (about two multiply-adds per SM and clock): the layout
// has to cut operations and keep warps full, nothing else matters much -- words
// of one form follow each other, so that a warp runs one operation on 32
// patterns.  Currents live in shared memory, or, where an event's do not fit
// (two quark lines with three gluons), in a region of global memory per CTA that
// stays in L2; the amplitudes likewise (gg>5g).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "amp_common.cuh"
#include "kernels.h"
#include "ordered_eval.cuh"

namespace mea {
namespace {

constexpr int kOrdThreads = 256;

// Shares of the colour matrix' rows that different threads sum.
__host__ __device__ __forceinline__ int ord_shares(int n_colour) { return n_colour > 64 ? 8 : n_colour > 16 ? 4 : 1; }

// Shared memory per event: event table, |M_h|^2 shares, currents and amplitudes where they fit.
__host__ __device__ __forceinline__ size_t ord_event_bytes(const DevProgram& p, bool area, bool amps) {
  size_t b = (size_t)event_table_stride(p.n_ext, p.n_masks) * 8;
  b += (size_t)p.ord_H * ord_shares(p.ord_colour) * 8;
  if (area) b += (size_t)p.ord_area * 8;
  if (amps) b += (size_t)p.ord_nf * 16;
  return (b + 15) & ~size_t(15);
}
__host__ __device__ __forceinline__ size_t ord_smem(const DevProgram& p, int E, bool area, bool amps) {
  return ord_event_bytes(p, area, amps) * E + 4 * (size_t)E + 16;
}

__global__ void __launch_bounds__(kOrdThreads) ordered_kernel(const DevProgram P, const AmpLaunch A, const int E,
                                                              const bool area_smem, const bool amps_smem) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int t = threadIdx.x, L = blockDim.x;
  const int tab_stride = event_table_stride(P.n_ext, P.n_masks);
  const int H = P.ord_H, m = P.ord_colour, NS = ord_shares(m);
  // currents first (16-byte accesses), then amplitudes, tables, results
  unsigned char* at = smem;
  double *area, *amps;
  if (area_smem) { area = reinterpret_cast<double*>(at); at += (size_t)E * P.ord_area * 8; }
  else area = reinterpret_cast<double*>(A.slot_scratch) + (size_t)blockIdx.x * E * P.ord_area;
  if (amps_smem) { amps = reinterpret_cast<double*>(at); at += (size_t)E * P.ord_nf * 16; }
  else amps = reinterpret_cast<double*>(A.jamp_scratch) + (size_t)blockIdx.x * E * P.ord_nf * 2;
  double* tab = reinterpret_cast<double*>(at);
  at += (size_t)E * tab_stride * 8;
  double* res = reinterpret_cast<double*>(at);
  at += (size_t)E * H * NS * 8;
  unsigned int* evflag = reinterpret_cast<unsigned int*>(at);
  for (int i = t; i < E; i += L) evflag[i] = 0u;

  const bool listed = A.event_list != nullptr;
  const int64_t n = listed ? (int64_t)(*A.list_count) : A.n_events;
  const int64_t n_tiles = (n + E - 1) / E;
  const double scale = P.ord_norm;
  AmpLaunch fin = A;
  fin.paired = false;  // the recursion's combinations carry the factor of their flipped ones

  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t ev0 = tile * E;
    const int here = (int)(n - ev0 < E ? n - ev0 : E);
    __syncthreads();
    tile_prep<double>(P, A, tab, tab_stride, ev0, n, E, t, L, evflag);
    __syncthreads();
    for (int s = 0; s < P.ord_n_stages; ++s) {
      const OrdStage st = P.ord_stages[s];
      const int items = (int)st.words << st.nb;
      for (int i = t; i < here * items; i += L) {
        const int e = i / items, q = i - e * items;
        OrdEvent ev;
        ev.area = area + (size_t)e * P.ord_area;
        ev.F = amps + (size_t)e * P.ord_nf * 2;
        ev.et = tab + (size_t)e * tab_stride;
        ev.mt = ev.et + 8 * P.n_ext;
        ev.leg = P.leg_info;
        ord_item(st, P.ord_rec + st.rec + (size_t)(q >> st.nb) * st.stride, (uint32_t)q & ((1u << st.nb) - 1u), ev);
      }
      if (P.ord_barrier[s]) __syncthreads();
    }
    // colour sum: rows a = share, share + NS, ... of the upper triangle
    // (off-diagonal entries doubled)
    for (int i = t; i < here * H * NS; i += L) {
      const int e = i / (H * NS), q = i - e * (H * NS), sh = q / H, h = q - sh * H;
      const double2* F = reinterpret_cast<const double2*>(amps + (size_t)e * P.ord_nf * 2);
      const uint16_t* ix = P.ord_fidx + h;
      const int a0 = P.ord_range[2 * h], a1 = P.ord_range[2 * h + 1];
      double tot = 0.0;
      for (int a = a0 + sh; a < a1; a += NS) {
        const double* k = P.ord_k + (size_t)a * m;
        const double2 x = F[__ldg(ix + a * H)];
        double zr = k[a] * x.x, zi = k[a] * x.y;
        for (int b = a + 1; b < a1; ++b) {
          const double2 y = F[__ldg(ix + b * H)];
          const double kb = __ldg(k + b);
          zr += kb * y.x;
          zi += kb * y.y;
        }
        tot += x.x * zr + x.y * zi;
      }
      const double v = scale * tot;
      res[(size_t)e * H * NS + sh * H + h] = isfinite(v) ? v : __longlong_as_double(0x7ff8000000000000ll);
    }
    __syncthreads();
    tile_finish<false>(fin, t, E, H * NS, ev0, n, listed, res, reinterpret_cast<const float*>(res), evflag);
  }
}

}  // namespace

bool ordered_supported(const DevProgram& p, bool fp64, int H) { return fp64 && p.ord_stages != nullptr && H == p.ord_lanes; }

// Tiles worth timing.  Everything of an event in shared memory where it fits
// with the others of its tile, else one event per CTA with the amplitudes, then
// the currents, in global memory.
std::vector<AmpConfig> ordered_candidates(const DevProgram& p, int H, int num_sms, size_t max_smem, size_t smem_per_sm) {
  std::vector<AmpConfig> out;
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, (const void*)ordered_kernel) != cudaSuccess) {
    cudaGetLastError();
    return out;
  }
  const int regs_warp = ((std::max(fa.numRegs, 1) + 7) / 8) * 8 * 32;
  auto add = [&](int E, int threads, bool area, bool amps) {
    const size_t sm = ord_smem(p, E, area, amps);
    if (sm > max_smem) return false;
    const int res = std::min({65536 / (regs_warp * (threads / 32)), (int)(smem_per_sm / (sm + 1024)), 2048 / threads, 32});
    if (res < 1) return false;
    AmpConfig c;
    c.ordered = true;
    c.H = H;
    c.E_cta = E;
    c.threads = threads;
    c.smem = sm;
    c.slots_in_smem = area;
    c.jamp_in_smem = amps;
    c.per_sm = res;
    c.grid = res * num_sms;
    out.push_back(c);
    return true;
  };
  bool any = false;
  for (int E : {1, 2, 4, 8, 16, 32, 64})
    for (int threads : {128, 256}) any = add(E, threads, true, true) || any;
  if (!any && !add(1, 256, true, false)) add(1, 256, false, false);
  return out;
}

// Untuned: enough events that a stage of a dozen patterns per event fills the
// CTA, with at least two CTAs per SM.
const AmpConfig* ordered_default(const std::vector<AmpConfig>& cands) {
  const AmpConfig* best = &cands.front();
  for (const AmpConfig& c : cands)
    if (c.E_cta <= 32 && c.per_sm >= std::min(2, best->per_sm) && c.per_sm * c.threads >= std::min(512, best->per_sm * best->threads) &&
        (c.E_cta > best->E_cta || (c.E_cta == best->E_cta && c.threads > best->threads)))
      best = &c;
  return best;
}

size_t ordered_area_bytes(const DevProgram& p, const AmpConfig& c) {
  return c.slots_in_smem ? 0 : (size_t)c.grid * c.E_cta * p.ord_area * 8;
}
size_t ordered_amp_bytes(const DevProgram& p, const AmpConfig& c) {
  return c.jamp_in_smem ? 0 : (size_t)c.grid * c.E_cta * p.ord_nf * 16;
}

cudaError_t launch_ordered(const DevProgram& p, const AmpConfig& c, const AmpLaunch& a, cudaStream_t s) {
  if (!ordered_supported(p, true, c.H) || a.hel_mode != 0 || a.amp_out) return cudaErrorInvalidValue;
  if (c.threads < 32 || c.threads > kOrdThreads || c.threads % 32 != 0 || c.E_cta < 1 ||
      c.smem != ord_smem(p, c.E_cta, c.slots_in_smem, c.jamp_in_smem) || (!c.slots_in_smem && !a.slot_scratch) ||
      (!c.jamp_in_smem && !a.jamp_scratch))
    return cudaErrorInvalidConfiguration;
  // fewer events than the tiles of a full grid hold: smaller tiles on more CTAs
  int E = c.E_cta, grid = c.grid;
  if (!a.event_list && c.slots_in_smem && c.jamp_in_smem) {
    const int64_t full = (int64_t)c.per_sm * p.num_sms;
    E = (int)std::max<int64_t>(1, std::min<int64_t>(E, (a.n_events + full - 1) / full));
    grid = (int)std::min<int64_t>(full, (a.n_events + E - 1) / E);
  }
  cudaError_t e = ensure_dynamic_smem((const void*)ordered_kernel, c.smem);
  if (e != cudaSuccess) return e;
  if (cudaFuncSetAttribute(ordered_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, carveout_percent(p, c)) != cudaSuccess)
    cudaGetLastError();
  ordered_kernel<<<grid, c.threads, ord_smem(p, E, c.slots_in_smem, c.jamp_in_smem), s>>>(p, a, E, c.slots_in_smem, c.jamp_in_smem);
  return cudaGetLastError();
}

}  // namespace mea
