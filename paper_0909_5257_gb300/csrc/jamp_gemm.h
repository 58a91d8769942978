// Colour amplitudes from Feynman-diagram amplitudes on the tensor cores.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "colour_base.h"
#include "generator.h"

namespace mea {

// Host-side description of the diagram -> colour-amplitude map
// J_alpha = sum_d c_{alpha d} A_d of a program (Eq. (color-amplitude)), with
// every coefficient real: c = cfac * n, n a small integer.
//
// Only a base of mb of the m colour amplitudes is contracted where the others
// are signed sums of it (the Kleiss-Kuijf relations of the gluon processes,
// found and checked here on the integer coefficients: n_alpha d = sum_b
// +-n_b d for every diagram); otherwise mb = m.  The base is split into
// n_splits column blocks of nc; the diagrams are stored in the order row[],
// sorted by the splits they touch, and a split's chunks without any of its
// coefficients are left out.
struct JampMap {
  bool ok = false;          // false: some coefficient is not real (path unavailable)
  int kd = 0;               // diagrams (K)
  int m = 0;                // colour amplitudes
  int mb = 0;               // of them contracted (the base: columns 0 .. mb - 1)
  int nc = 0;               // base columns per CTA (multiple of 16, 3 * nc <= 512)
  int n_splits = 0;         // ceil(mb / nc)
  int q = 0;                // digit bound 2^q (see jamp_gemm.cu)
  double cfac = 1;          // common factor of the coefficients
  std::vector<__half> tiles;  // per listed chunk [nc x 64] canonical K-major fp16 tiles of -n
  std::vector<int> chunks;    // chunk (64 consecutive rows) of every tile, split by split
  std::vector<int> split_begin;  // [n_splits + 1] into chunks
  std::vector<int> row;       // [kd] row of diagram d in the amplitude buffer
  std::vector<float> weight;  // [kd] sum_alpha |c_{alpha d}| (cancellation indicator)
  // m > mb: colour amplitudes mb .. m - 1 as sums of base ones: for each the
  // begin, the first subtracted and the end term in kk_term
  std::vector<uint16_t> kk_index;  // [3 * (m - mb)]
  std::vector<uint16_t> kk_term;
};

// base: find_colour_base(p), found here when null
JampMap build_jamp_map(const Program& p, const ColourBase* base = nullptr);

// `ops` (all amplitudes of the program, in its order) with every amplitude's row
// and weight bits in its colour fields (DevProgram::ops_out).
std::vector<Op> amplitude_output_ops(std::vector<Op> ops, const JampMap& m);

struct JampGemmArgs {
  const float* A = nullptr;      // [kd][lda]: A[d*lda + 2p] = Re A_d, [.. + 1] = Im A_d of pair p
  int64_t lda = 0;
  const float* rowmax = nullptr;  // [2*n_pairs] max_d |A| of each row (NaN when a row is not finite)
  int64_t n_pairs = 0;
  int kd = 0, m = 0, mb = 0, nc = 0, n_splits = 0, q = 0;
  double cfac = 1;
  const __half* tiles = nullptr;  // device copies of JampMap::tiles, chunks, split_begin
  const int* chunks = nullptr;
  const int* split_begin = nullptr;
  int n_chunks = 0;               // listed chunks of all splits
  const uint16_t* kk_index = nullptr;  // m > mb: device copies of JampMap::kk_index, kk_term
  const uint16_t* kk_term = nullptr;
  int kk_terms = 0;
  float* J = nullptr;             // [2*n_pairs][ldj] output rows (re, im) per pair
  int ldj = 0;
  float* jabs = nullptr;          // [n_splits][n_pairs]: sum |J| over the split's columns
  int* status = nullptr;          // set to 1 when a bounded wait expired
  uint32_t spin_limit = 1u << 19;  // polls of the issuing thread's waits, tc::kSpinLimit (a test makes them run out)
};

cudaError_t launch_jamp_gemm(const JampGemmArgs& a, int num_sms, cudaStream_t s);

}  // namespace mea
