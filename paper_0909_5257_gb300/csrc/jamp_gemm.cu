// Colour amplitudes J_alpha = sum_d c_{alpha d} A_d (Eq. (color-amplitude))
// as an exact integer contraction on the tensor cores.
//
// The amplitude kernel writes every Feynman-diagram amplitude A_d of every
// (event, helicity) pair in FP32.  All colour coefficients of the processes
// handled here are real, c = cfac * n with small integers n.  Per row r (the
// real or the imaginary parts of one pair) the amplitudes are scaled by a
// power of two, x = A * 2^(q - e_r) with 2^(e_r - 1) <= max_d |A_rd| < 2^e_r,
// so that |x| < 2^q, and split into three integer digits
//     x = h + m 2^-(q+1) + l 2^-2(q+1) + O(2^-(2q+3)),   |h|, |m|, |l| <= 2^q,
// each exact in FP16 (q <= 11).  tcgen05.mma kind::f16 then forms
// H = sum_d n_d h_d, M = sum_d n_d m_d, L = sum_d n_d l_d in three FP32
// tensor-memory accumulators over the whole diagram sum: every product and
// every partial sum is an integer below sum_d |n_{alpha d}| 2^q < 2^24, so the
// accumulation is exact whatever order or internal rounding the tensor core
// uses.  The epilogue recombines cfac * 2^(e_r - q) (H + M 2^-(q+1) +
// L 2^-2(q+1)) with two FP32 FMAs (within an ulp of the exact value).  The
// only other error is the digit truncation, below 2^-(3q+3) of the row
// maximum: the colour amplitudes come out as the FP32-rounded exact sum of the
// FP32 diagram amplitudes (the compensated summation of the paper's Sec. 3.2
// step 3 with nothing left to compensate).
//
// Base.  Where colour amplitudes are signed sums of others (gluon processes:
// (n-2)! of the (n-1)!/2 orderings by the Kleiss-Kuijf relations; 120 of 360
// for gg>5g), only the base is contracted: H, M and L of the others are the
// same sums of the base's H, M and L, formed as 32-bit integers, so every
// result is that of contracting all columns, bit for bit -- while one column
// block fits the tensor memory instead of three and every amplitude is read
// and split into digits once instead of three times.
//
// Tile: 128 rows x nc columns, K in chunks of 64 diagrams; rows 0..63 are the
// real and 64..127 the imaginary parts of 64 pairs, so that a thread reads a
// pair's (Re, Im) in one 8-byte load and converts both with packed FP32 pairs
// (4 two-lane operations per element instead of 8).  Sixteen warps convert
// into two shared-memory stages, a seventeenth issues the MMAs and the bulk
// copies of the coefficient tiles (four stages); they meet at mbarriers, never
// at a CTA barrier inside the loop, and the loads run two chunks ahead across
// tile boundaries.
//
// Every mbarrier wait is bounded.  A wait that expires records an error in
// *status and sets a flag that ends the others' waits.  Barriers have no bound, so
// nobody may leave one that others stand at: a wait's outcome is made uniform
// over its warp, and after the waits of a tile all converters meet at one
// barrier that also votes -- each reaches it once per tile, whatever its waits
// gave, and they go on or leave together.  The issuing thread, on every path,
// waits (with a bound) for the copies and MMAs it has issued before the CTA's
// shared and tensor memory go away.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <numeric>

#include "jamp_gemm.h"
#include "kernels.h"
#include "tc_common.cuh"

namespace mea {
namespace {

using namespace tc;

constexpr int kConvert = 512;            // 16 warps convert and run the epilogue
constexpr int kThreads = kConvert + 32;  // and one issues copies and MMAs
constexpr int kM = 128;
constexpr int kPairs = kM / 2;
constexpr int kKC = 64;
constexpr int kBStages = 4;
constexpr int kStageA = kM * kKC * 2;       // one FP16 digit plane of A
constexpr float kRoundMagic = 12582912.0f;  // 1.5 * 2^23
constexpr int kMaxNC = 128;                 // 3 accumulators of nc columns in 512 TMEM columns

// two FP32 values operated on together
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ void bar_converters() { asm volatile("bar.sync 1, %0;" ::"n"(kConvert) : "memory"); }
// the same barrier; true where `ok` is on all of them
__device__ __forceinline__ bool vote_converters(bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r)
      : "r"((uint32_t)ok), "n"(kConvert)
      : "memory");
  return r != 0;
}

__host__ __device__ constexpr size_t tail_bytes() {
  // 2 + 2 + kBStages + 1 barriers, TMEM slot and abort flag, [kM] row scales, [8][kM] partial sums of |J|
  return 128 + (size_t)kM * 4 + (size_t)8 * kM * 4;
}

// The CTA's sequence of (tile, split) works and their chunks: work w = tile *
// n_splits + split for w = blockIdx.x, + gridDim.x, ...
struct Walk {
  int tile, split, c;         // c: index into the chunk list, within the split's part of it
  __device__ __forceinline__ void start(int n_splits, const int* begin) {
    tile = (int)blockIdx.x / n_splits;
    split = (int)blockIdx.x - tile * n_splits;
    c = begin[split];
  }
  __device__ __forceinline__ void next_work(int n_splits, const int* begin, int d_tile, int d_split) {
    tile += d_tile;
    split += d_split;
    if (split >= n_splits) {
      split -= n_splits;
      ++tile;
    }
    c = begin[split];
  }
  __device__ __forceinline__ void next_chunk(int n_splits, const int* begin, int d_tile, int d_split) {
    if (++c >= begin[split + 1]) next_work(n_splits, begin, d_tile, d_split);
  }
};

__global__ void __launch_bounds__(kThreads, 1) jamp_gemm_kernel(JampGemmArgs g) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int t = threadIdx.x;
  const int warp = t >> 5;
  const int NC = g.nc;
  const uint32_t b_bytes = (uint32_t)(NC * kKC * 2);
  unsigned char* b_base = smem + 2 * 3 * kStageA;
  unsigned char* tail = b_base + (size_t)kBStages * b_bytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(tail);  // [2] digits of a stage written (16 warps)
  uint64_t* empty = full + 2;                          // [2] MMAs of a stage done
  uint64_t* bfull = empty + 2;                         // [kBStages] coefficient tile landed
  uint64_t* done = bfull + kBStages;                   // MMAs of a tile done
  uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  float* rscale = reinterpret_cast<float*>(tail + 128);  // [kM]
  float* rowabs = rscale + kM;                           // [8][kM]
  int* begin = reinterpret_cast<int*>(rowabs + 8 * kM);  // [n_splits + 1]
  int* chunks = begin + g.n_splits + 1;                  // [n_chunks]
  uint16_t* kk_index = reinterpret_cast<uint16_t*>(chunks + g.n_chunks);
  const int n_kk = g.m - g.mb;
  uint16_t* kk_term = kk_index + 3 * n_kk;

  uint32_t tmem_cols = 32;
  while (tmem_cols < (uint32_t)(3 * NC)) tmem_cols <<= 1;
  if (t == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&full[s], kConvert / 32);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < kBStages; ++s) mbar_init(&bfull[s], 1);
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *abort_flag = 0;
  }
  for (int i = t; i <= g.n_splits; i += kThreads) begin[i] = g.split_begin[i];
  for (int i = t; i < g.n_chunks; i += kThreads) chunks[i] = g.chunks[i];
  for (int i = t; i < 3 * n_kk; i += kThreads) kk_index[i] = g.kk_index[i];
  for (int i = t; i < g.kk_terms; i += kThreads) kk_term[i] = g.kk_term[i];
  if (warp == 0) tmem_alloc(tslot, tmem_cols);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;
  const uint32_t d_h = tmem, d_m = tmem + (uint32_t)NC, d_l = tmem + (uint32_t)(2 * NC);

  const int n_tiles = (int)((g.n_pairs + kPairs - 1) / kPairs), ns = g.n_splits;
  const int d_tile = (int)gridDim.x / ns, d_split = (int)gridDim.x - d_tile * ns;
  auto expired = [&]() {
    *abort_flag = 1;
    if (g.status) atomicExch(g.status, 1);
  };

  if (warp == kConvert / 32) {
    // ---- copies and MMAs: one thread
    if ((t & 31) == 0) {
      const uint32_t idesc = make_idesc(kM, NC);
      uint32_t issued = 0, i = 0;  // coefficient copies issued, chunks contracted
      bool ok = true;
      Walk ahead, w;
      ahead.start(ns, begin);
      auto copy = [&]() {  // the coefficient tile of `ahead` into stage issued % kBStages
        if (ahead.tile >= n_tiles) return;
        uint64_t* bar = &bfull[issued % kBStages];
        mbar_expect_tx(bar, b_bytes);
        bulk_g2s(b_base + (size_t)(issued % kBStages) * b_bytes, g.tiles + (size_t)ahead.c * NC * kKC, b_bytes, bar);
        ++issued;
        ahead.next_chunk(ns, begin, d_tile, d_split);
      };
      for (int k = 0; k < kBStages - 2; ++k) copy();
      for (w.start(ns, begin); w.tile < n_tiles && ok; w.next_work(ns, begin, d_tile, d_split)) {
        const int n_kc = begin[w.split + 1] - begin[w.split];
        for (int kc = 0; kc < n_kc && ok; ++kc, ++i) {
          const int st = (int)(i & 1u);
          // the digits of chunk i (then the MMAs of chunk i - 2 are done too:
          // the converters waited for them before they wrote)
          ok = mbar_wait_abort(&full[st], (i >> 1) & 1u, abort_flag, g.spin_limit) &&
               mbar_wait_abort(&bfull[i % kBStages], (i / kBStages) & 1u, abort_flag, g.spin_limit);
          if (!ok) break;
          copy();  // chunk i + 2 into the coefficient stage chunk i - 2 read
          fence_after();
          const uint32_t lbo = 128, sbo = (kKC / 8) * 128;
          const uint32_t a_h = smem_u32(smem + (size_t)st * 3 * kStageA);
          const uint32_t b_t = smem_u32(b_base + (size_t)(i % kBStages) * b_bytes);
#pragma unroll
          for (int ks = 0; ks < kKC / 16; ++ks) {
            const uint32_t koff = (uint32_t)(ks * 2 * 128);
            const uint64_t db = make_desc(b_t + koff, lbo, sbo);
            const uint32_t acc = (kc > 0 || ks > 0) ? 1u : 0u;
            mma_f16(d_l, make_desc(a_h + 2 * kStageA + koff, lbo, sbo), db, idesc, acc);
            mma_f16(d_m, make_desc(a_h + kStageA + koff, lbo, sbo), db, idesc, acc);
            mma_f16(d_h, make_desc(a_h + koff, lbo, sbo), db, idesc, acc);
          }
          mma_commit(&empty[st]);
          if (kc == n_kc - 1) mma_commit(done);
        }
      }
      if (!ok) expired();
      // copies in flight land, and the MMAs issued finish, before the CTA's shared
      // and tensor memory go away (also where only converters gave up)
      for (uint32_t k = i; k < issued; ++k) mbar_wait(&bfull[k % kBStages], (k / kBStages) & 1u);
      for (uint32_t k = i > 2 ? i - 2 : 0; k < i; ++k) mbar_wait(&empty[k & 1u], (k >> 1) & 1u);
    }
    __syncwarp();
  } else {
    // ---- digits: thread -> (pair, 8 consecutive diagrams)
    const int p = t & (kPairs - 1), kg = t >> 6;
    const float w1 = ldexpf(1.f, g.q + 1);  // digit base
    const float inv_w1 = 1.f / w1, inv_w2 = inv_w1 * inv_w1;  // powers of two
    const uint64_t M2 = pack2(kRoundMagic, kRoundMagic), nM2 = pack2(-kRoundMagic, -kRoundMagic);
    const uint64_t w2 = pack2(w1, w1), nw2 = pack2(-w1, -w1);
    typedef uint64_t ABuf[8];  // (Re, Im) of 8 diagrams
    ABuf pa0, pa1;             // chunks two apart: each is loaded two chunks ahead
    auto prefetch = [&](const Walk& it, ABuf& pa) {
      const int64_t pair = (int64_t)it.tile * kPairs + p;
      if (pair < g.n_pairs) {
        const int d0 = chunks[it.c] * kKC + kg * 8;
        const float* src = g.A + (size_t)d0 * g.lda + 2 * pair;
        if (d0 + 8 <= g.kd) {
#pragma unroll
          for (int i = 0; i < 8; ++i) pa[i] = __ldg(reinterpret_cast<const unsigned long long*>(src + (size_t)i * g.lda));
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i)
            pa[i] = d0 + i < g.kd ? __ldg(reinterpret_cast<const unsigned long long*>(src + (size_t)i * g.lda)) : 0ull;
        }
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) pa[i] = 0ull;
      }
    };
    auto scale_of = [&](float mx) {
      if (!isfinite(mx)) return __int_as_float(0x7fc00000);  // a non-finite row stays non-finite (flagged later)
      int e = 0;
      if (mx > 0.f) frexpf(mx, &e);
      return ldexpf(1.f, max(-120, min(120, g.q - e)));
    };
    auto row_max = [&](int tile) {  // of this thread's pair
      const int64_t pair = (int64_t)tile * kPairs + p;
      return pair < g.n_pairs ? __ldg(reinterpret_cast<const float2*>(g.rowmax) + pair) : make_float2(0.f, 0.f);
    };
    // a bounded wait with one outcome for the warp (its limit is a constant: read from
    // the launch arguments it costs the conversion registers, 2 to 4 % of the stage)
    auto wait = [&](uint64_t* bar, uint32_t phase) {
      return __all_sync(0xffffffffu, mbar_wait_abort(bar, phase, abort_flag)) != 0;
    };
    uint32_t i = 0, tile_no = 0;
    Walk ahead, w, w_next;
    ahead.start(ns, begin);
    prefetch(ahead, pa0);
    ahead.next_chunk(ns, begin, d_tile, d_split);
    prefetch(ahead, pa1);
    ahead.next_chunk(ns, begin, d_tile, d_split);
    w.start(ns, begin);
    float2 mx = row_max(w.tile);
    for (; w.tile < n_tiles; w = w_next, ++tile_no) {
      const float s_re = scale_of(mx.x), s_im = scale_of(mx.y);
      w_next = w;
      w_next.next_work(ns, begin, d_tile, d_split);
      mx = row_max(w_next.tile);
      const uint64_t s2 = pack2(s_re, s_im), ns2 = pack2(-s_re, -s_im);
      if (kg == 0) {  // read by the epilogue, behind its barrier
        rscale[p] = s_re;
        rscale[kPairs + p] = s_im;
      }
      const int n_kc = begin[w.split + 1] - begin[w.split];
      auto step = [&](ABuf& pa) {
        const int st = (int)(i & 1u);
        if (i >= 2 && !wait(&empty[st], ((i - 2) >> 1) & 1u)) return false;
        unsigned char* a_h = smem + (size_t)st * 3 * kStageA;
        // x = a s, r1 = (x - h) w, r2 = (r1 - m) w: every product by the powers
        // of two s and w and every difference of a value and its nearest
        // integer is exact, so each FMA rounds once, where adding 1.5 * 2^23
        // rounds to the nearest integer.  The digits are formed negated (the
        // packed operations have no negation): -h = (a (-s) - M) + M; the
        // coefficient tiles hold -n.
        __align__(16) __half2 hr[4], hi[4], mr[4], mi[4], lr[4], li[4];
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
          float h[2][2], m[2][2], l[2][2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const uint64_t a = pa[k + u];
            const uint64_t nh = add2(fma2(a, ns2, nM2), M2);
            const uint64_t y1 = fma2(a, s2, nh);
            const uint64_t nm = add2(fma2(y1, nw2, nM2), M2);
            const uint64_t y2 = fma2(y1, w2, nm);
            const uint64_t nl = add2(fma2(y2, nw2, nM2), M2);
            unpack2(nh, h[u][0], h[u][1]);
            unpack2(nm, m[u][0], m[u][1]);
            unpack2(nl, l[u][0], l[u][1]);
          }
          // integers of at most 2^q <= 2048 in magnitude: exact in FP16
          hr[k / 2] = __floats2half2_rn(h[0][0], h[1][0]);
          hi[k / 2] = __floats2half2_rn(h[0][1], h[1][1]);
          mr[k / 2] = __floats2half2_rn(m[0][0], m[1][0]);
          mi[k / 2] = __floats2half2_rn(m[0][1], m[1][1]);
          lr[k / 2] = __floats2half2_rn(l[0][0], l[1][0]);
          li[k / 2] = __floats2half2_rn(l[0][1], l[1][1]);
        }
        const uint32_t off_r = canon_off(p, kg * 8, kKC), off_i = canon_off(kPairs + p, kg * 8, kKC);
        *reinterpret_cast<uint4*>(a_h + off_r) = *reinterpret_cast<const uint4*>(hr);
        *reinterpret_cast<uint4*>(a_h + off_i) = *reinterpret_cast<const uint4*>(hi);
        *reinterpret_cast<uint4*>(a_h + kStageA + off_r) = *reinterpret_cast<const uint4*>(mr);
        *reinterpret_cast<uint4*>(a_h + kStageA + off_i) = *reinterpret_cast<const uint4*>(mi);
        *reinterpret_cast<uint4*>(a_h + 2 * kStageA + off_r) = *reinterpret_cast<const uint4*>(lr);
        *reinterpret_cast<uint4*>(a_h + 2 * kStageA + off_i) = *reinterpret_cast<const uint4*>(li);
        prefetch(ahead, pa);
        ahead.next_chunk(ns, begin, d_tile, d_split);
        fence_async_smem();
        fence_before();
        __syncwarp();
        if ((t & 31) == 0) mbar_arrive(&full[st]);
        ++i;
        return true;
      };
      // the buffers alternate over all chunks of the CTA (i even: pa0)
      bool ok = true;
      int kc = 0;
      if (i & 1u) {
        ok = step(pa1);
        kc = 1;
      }
      for (; ok && kc + 1 < n_kc; kc += 2) ok = step(pa0) && step(pa1);
      if (ok && kc < n_kc) ok = step(pa0);
      ok = ok && wait(done, tile_no & 1u);
      if (!ok) expired();
      if (!vote_converters(ok)) break;  // also: row scales written
      fence_after();

      // ---- epilogue: warp -> tensor-memory lanes 32 (warp mod 4) .., a quarter of the columns
      const int64_t mt = w.tile;
      const int split = w.split;
      const int n0 = split * NC;
      const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;
      const int lrow = (warp & 3) * 32 + (t & 31);
      const int quarter = warp >> 2;
      if (n_kk == 0) {
        const int64_t pair = mt * kPairs + (lrow & (kPairs - 1));
        const float back = (float)g.cfac / rscale[lrow];  // cfac (1 or 2) times a power of two
        float* jrow = g.J + (size_t)(2 * pair + (lrow >> 6)) * g.ldj;
        float sabs = 0.f;
        for (int c0 = 16 * quarter; c0 < NC && n0 + c0 < g.mb; c0 += 64) {
          float vh[16], vm[16], vl[16];
          tmem_ld16(d_h + lane + (uint32_t)c0, vh);
          tmem_ld16(d_m + lane + (uint32_t)c0, vm);
          tmem_ld16(d_l + lane + (uint32_t)c0, vl);
          if (pair < g.n_pairs) {
            float v[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              // h + m/2^(q+1) + l/2^2(q+1): the inner FMA is exact up to one rounding and the
              // l term lies below the last digit of m, so v is within an ulp of the exact sum
              v[k] = fmaf(vl[k], inv_w2, fmaf(vm[k], inv_w1, vh[k])) * back;
              if (n0 + c0 + k < g.mb) sabs += fabsf(v[k]);
            }
            // rows of J are 16-byte aligned (ldj is a multiple of 16) and the
            // last block of 16 columns ends within ldj: whole vectors, zeros beyond m
            float4* dst = reinterpret_cast<float4*>(jrow + n0 + c0);
#pragma unroll
            for (int k = 0; k < 4; ++k) dst[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
          }
        }
        rowabs[quarter * kM + lrow] = sabs;
      } else {
        // H, M, L of the base as integers, [plane][column][64 rows] over the
        // digit stages (all their MMAs are done), for the real, then the
        // imaginary rows; then every thread sums columns of its row
        int* stage = reinterpret_cast<int*>(smem);
        const int64_t pair = mt * kPairs + p;
        for (int half = 0; half < 2; ++half) {
          if (half) bar_converters();  // the other half's sums are done
          if ((lrow >> 6) == half)
            for (int c0 = 16 * quarter; c0 < g.mb; c0 += 64) {
              float v[3][16];
              tmem_ld16(d_h + lane + (uint32_t)c0, v[0]);
              tmem_ld16(d_m + lane + (uint32_t)c0, v[1]);
              tmem_ld16(d_l + lane + (uint32_t)c0, v[2]);
#pragma unroll
              for (int k = 0; k < 16; ++k)
                if (c0 + k < g.mb)
#pragma unroll
                  for (int pl = 0; pl < 3; ++pl)
                    stage[(pl * g.mb + c0 + k) * kPairs + (lrow & (kPairs - 1))] = __float2int_rn(v[pl][k]);
            }
          bar_converters();
          const float back = (float)g.cfac / rscale[half * kPairs + p];
          float* jrow = g.J + (size_t)(2 * pair + half) * g.ldj;
          const int* col = stage + p;
          const int plane = g.mb * kPairs;
          float sabs = 0.f;
          for (int a0 = 8 * kg; a0 < g.m; a0 += 64) {
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const int a = a0 + k;
              int h = 0, m = 0, l = 0;
              if (a < g.mb) {
                h = col[a * kPairs];
                m = col[a * kPairs + plane];
                l = col[a * kPairs + 2 * plane];
              } else if (a < g.m) {
                const uint16_t* ix = kk_index + 3 * (a - g.mb);
                const int b1 = ix[1], b2 = ix[2];
                for (int b = ix[0]; b < b1; ++b) {
                  const int* c = col + kk_term[b] * kPairs;
                  h += c[0];
                  m += c[plane];
                  l += c[2 * plane];
                }
                for (int b = b1; b < b2; ++b) {
                  const int* c = col + kk_term[b] * kPairs;
                  h -= c[0];
                  m -= c[plane];
                  l -= c[2 * plane];
                }
              }
              v[k] = fmaf((float)l, inv_w2, fmaf((float)m, inv_w1, (float)h)) * back;
              if (a < g.m) sabs += fabsf(v[k]);
            }
            if (pair < g.n_pairs) {
              float4* dst = reinterpret_cast<float4*>(jrow + a0);
              dst[0] = make_float4(v[0], v[1], v[2], v[3]);
              dst[1] = make_float4(v[4], v[5], v[6], v[7]);
            }
          }
          rowabs[kg * kM + half * kPairs + p] = sabs;
        }
      }
      fence_before();
      bar_converters();  // sums written; tensor memory and stages read
      if (kg == 0 && g.jabs) {
        const int64_t pair = mt * kPairs + p;
        float s = 0.f;
        for (int k = 0; k < (n_kk == 0 ? 4 : 8); ++k) s += rowabs[k * kM + p] + rowabs[k * kM + kPairs + p];
        if (pair < g.n_pairs) g.jabs[(size_t)split * g.n_pairs + pair] = s;
      }
      bar_converters();  // row scales and sums free for the next tile
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) tmem_dealloc(tmem, tmem_cols);
}

}  // namespace

JampMap build_jamp_map(const Program& p, const ColourBase* known) {
  JampMap M;
  M.m = p.n_jamp;
  int kd = 0;
  int g = 0;
  bool real = true;
  for (const Op& op : p.ops) {
    if (!is_amp_op(op.type)) continue;
    ++kd;
    for (uint32_t k = 0; k < op.col_count; ++k) {
      const ColEntry& c = p.col[op.col_begin + k];
      if (c.im != 0) real = false;
      g = std::gcd(g, std::abs((int)c.re));
    }
  }
  M.kd = kd;
  if (!real || kd == 0 || M.m <= 0 || g == 0) return M;
  M.cfac = g;
  std::vector<int> C((size_t)M.m * kd, 0), colw(M.m, 0);
  M.weight.assign(kd, 0.f);
  int d = 0;
  for (const Op& op : p.ops) {
    if (!is_amp_op(op.type)) continue;
    for (uint32_t k = 0; k < op.col_count; ++k) {
      const ColEntry& c = p.col[op.col_begin + k];
      const int n = (amp_negated(op) ? -c.re : c.re) / g;
      colw[c.alpha] += std::abs(n);
      M.weight[d] += (float)std::abs((int)c.re);
      C[(size_t)c.alpha * kd + d] += n;
    }
    ++d;
  }
  const int wmax = *std::max_element(colw.begin(), colw.end());
  // exact accumulation: sum_d |n_{alpha d}| 2^q < 2^24 for every alpha, and 2^q <= 2048 (FP16 integers)
  int q = 11;
  while (q > 0 && (double)wmax * std::ldexp(1.0, q) >= 16777216.0) --q;
  M.q = q;

  // base columns: one block of them, their terms and a 64-row stage of their
  // integers must fit (kMaxNC columns do)
  const ColourBase base = known ? *known : find_colour_base(p);
  M.mb = M.m;
  if (base.mb < M.m && base.mb <= kMaxNC && base.term.size() <= 4096) {
    M.mb = base.mb;
    M.kk_index = base.index;
    M.kk_term = base.term;
  }
  M.nc = std::min(kMaxNC, ((M.mb + 15) / 16) * 16);
  M.n_splits = (M.mb + M.nc - 1) / M.nc;
  // balance the splits: the smallest multiple of 16 that still needs n_splits
  M.nc = std::min(M.nc, (((M.mb + M.n_splits - 1) / M.n_splits) + 15) / 16 * 16);

  // rows: diagrams sorted by the splits they touch
  std::vector<uint32_t> touch(kd, 0);
  for (int a = 0; a < M.mb; ++a)
    for (int x = 0; x < kd; ++x)
      if (C[(size_t)a * kd + x]) touch[x] |= 1u << std::min(31, a / M.nc);
  std::vector<int> order(kd);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return touch[a] < touch[b]; });
  M.row.assign(kd, 0);
  for (int r = 0; r < kd; ++r) M.row[order[r]] = r;
  const int n_kc = (kd + kKC - 1) / kKC;
  M.split_begin.push_back(0);
  for (int s = 0; s < M.n_splits; ++s) {
    for (int kc = 0; kc < n_kc; ++kc) {
      std::vector<__half> tile((size_t)M.nc * kKC, __float2half(0.f));
      bool any = false;
      for (int k = 0; k < kKC && kc * kKC + k < kd; ++k)
        for (int c = 0; c < M.nc && s * M.nc + c < M.mb; ++c) {
          const int n = C[(size_t)(s * M.nc + c) * kd + order[kc * kKC + k]];
          if (!n) continue;
          any = true;
          // every tile entry must itself be a small integer (coefficients of one diagram in one colour add up)
          if (std::abs(n) > 2048) return M;
          tile[tc::canon_off(c, k, kKC) / 2] = __float2half((float)-n);
        }
      if (any || (kc == n_kc - 1 && (int)M.chunks.size() == M.split_begin.back())) {  // at least one chunk
        M.chunks.push_back(kc);
        M.tiles.insert(M.tiles.end(), tile.begin(), tile.end());
      }
    }
    M.split_begin.push_back((int)M.chunks.size());
  }
  M.ok = q >= 8;  // digit truncation below 2^-27 of the row maximum
  return M;
}

std::vector<Op> amplitude_output_ops(std::vector<Op> ops, const JampMap& m) {
  size_t d = 0;
  for (Op& op : ops) {
    if (!is_amp_op(op.type)) continue;
    op.col_begin = (uint32_t)m.row.at(d);
    std::memcpy(&op.col_count, &m.weight.at(d), sizeof op.col_count);
    ++d;
  }
  return ops;
}

size_t jamp_gemm_smem(const JampGemmArgs& a) {
  return (size_t)2 * 3 * kStageA + (size_t)kBStages * a.nc * kKC * 2 + tail_bytes() +
         (size_t)4 * (a.n_splits + 1 + a.n_chunks) + (size_t)2 * (3 * (a.m - a.mb) + a.kk_terms) + 16;
}

cudaError_t launch_jamp_gemm(const JampGemmArgs& a, int num_sms, cudaStream_t s) {
  static_assert(JampGemmArgs().spin_limit == kSpinLimit, "the default of a launch");
  if (a.n_pairs <= 0) return cudaSuccess;
  if (a.n_pairs > (int64_t)1 << 36) return cudaErrorInvalidValue;  // tile numbers are 32-bit
  if (a.nc < 16 || a.nc > kMaxNC || a.nc % 16 != 0 || a.mb > a.m || a.mb > a.nc * a.n_splits) return cudaErrorInvalidValue;
  // 8-byte loads of a pair's amplitudes and row maxima, 16-byte stores of J
  // rows in blocks of 16 columns; one column block where sums of it follow
  if (a.lda % 2 != 0 || (reinterpret_cast<uintptr_t>(a.A) & 7) != 0 || (reinterpret_cast<uintptr_t>(a.rowmax) & 7) != 0 ||
      (reinterpret_cast<uintptr_t>(a.J) & 15) != 0 || a.ldj % 16 != 0 || a.ldj < a.m ||
      (a.m > a.mb && (a.n_splits != 1 || a.mb > a.nc)))
    return cudaErrorInvalidValue;
  const size_t sm = jamp_gemm_smem(a);
  cudaError_t e = ensure_dynamic_smem((const void*)jamp_gemm_kernel, sm);
  if (e != cudaSuccess) return e;
  const int64_t work = ((a.n_pairs + kPairs - 1) / kPairs) * a.n_splits;
  const int grid = (int)std::min<int64_t>(work, (int64_t)num_sms);
  jamp_gemm_kernel<<<grid, kThreads, sm, s>>>(a);
  e = cudaGetLastError();
  if (e == cudaSuccess) ++launch_counter();
  return e;
}

}  // namespace mea
