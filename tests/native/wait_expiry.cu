// Bounded waits of the tensor-core GEMMs that run out.  For every process given on
// the command line the colour-amplitude GEMM and the colour-sum GEMM run on random
// diagram amplitudes with the usual limit, then with limits of 0 polls (the first wait
// of the threads that issue copies and MMAs expires at once, and the others give up
// where they stand), 1, 2, .. polls: each launch must end without an error, report
// an expiry in its status word or none, and leave the next launch with the
// usual limit to give the first one's results bit for bit.  Prints per process
// the launches with an expiry; exit status 1 on a fault.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "colour_gemm.h"
#include "generator.h"
#include "jamp_gemm.h"
#include "tc_common.cuh"

using namespace mea;

constexpr uint32_t kDefault = tc::kSpinLimit;

static int faults = 0;
static void need(bool ok, const char* what) {
  if (!ok && ++faults <= 20) std::printf("fault: %s\n", what);
}
static void ck(cudaError_t e, const char* what) {
  if (e == cudaSuccess) return;
  std::printf("%s: %s\n", what, cudaGetErrorString(e));
  std::exit(2);
}
template <typename T>
static T* up(const std::vector<T>& v) {
  void* d = nullptr;
  ck(cudaMalloc(&d, v.size() * sizeof(T) + 16), "cudaMalloc");
  if (!v.empty()) ck(cudaMemcpy(d, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice), "cudaMemcpy");
  return static_cast<T*>(d);
}

int main(int argc, char** argv) {
  int sms = 0;
  ck(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0), "device");
  {
    // a wait with the usual limit that nothing ends: seconds
    std::vector<int> status(1, 0);
    int* s = up(status);
    cudaEvent_t e0, e1;
    ck(cudaEventCreate(&e0), "event");
    ck(cudaEventCreate(&e1), "event");
    ck(cudaEventRecord(e0), "event");
    ck(launch_wait_probe(s, kDefault, nullptr), "launch");
    ck(cudaEventRecord(e1), "event");
    ck(cudaEventSynchronize(e1), "kernel");
    float ms = 0;
    ck(cudaEventElapsedTime(&ms, e0, e1), "event");
    ck(cudaMemcpy(status.data(), s, sizeof(int), cudaMemcpyDeviceToHost), "status");
    std::printf("bound %.0f ms\n", ms);
    need(status[0] == 1 && ms < 10000, "bound of a wait");
    cudaFree(s);
  }
  for (int arg = 1; arg < argc; ++arg) {
    std::vector<int> pdg;
    std::string s = argv[arg];
    for (size_t p = 0; p < s.size();) {
      size_t e = s.find(',', p);
      if (e == std::string::npos) e = s.size();
      pdg.push_back(std::atoi(s.substr(p, e - p).c_str()));
      p = e + 1;
    }
    const Program P = build_program(pdg);
    const JampMap M = build_jamp_map(P);
    need(M.ok, "coefficients");
    const ColourTiles T = build_colour_tiles(P.cf_jamp, P.n_jamp);
    const int64_t n = 64 * 3 * (int64_t)sms + 37;  // several tiles per CTA, a ragged last one
    const int64_t lda = (2 * n + 127) / 128 * 128;
    const int ldj = (P.n_jamp + 15) / 16 * 16;
    std::mt19937_64 rng(0x5eed + arg);
    std::normal_distribution<float> gauss;
    std::vector<float> A((size_t)M.kd * lda, 0.f), rowmax(2 * n, 0.f);
    for (int d = 0; d < M.kd; ++d)
      for (int64_t r = 0; r < 2 * n; ++r) {
        const float v = gauss(rng);
        A[(size_t)d * lda + r] = v;
        rowmax[r] = std::max(rowmax[r], std::fabs(v));
      }
    std::vector<float> J((size_t)2 * n * ldj), jabs((size_t)M.n_splits * n);
    std::vector<double> pv(n);
    std::vector<int> status(1, 0);
    JampGemmArgs g;
    g.A = up(A);
    g.lda = lda;
    g.rowmax = up(rowmax);
    g.n_pairs = n;
    g.kd = M.kd; g.m = M.m; g.mb = M.mb; g.nc = M.nc; g.n_splits = M.n_splits; g.q = M.q; g.cfac = M.cfac;
    g.tiles = up(M.tiles);
    g.chunks = up(M.chunks);
    g.split_begin = up(M.split_begin);
    g.n_chunks = (int)M.chunks.size();
    g.kk_index = up(M.kk_index);
    g.kk_term = up(M.kk_term);
    g.kk_terms = (int)M.kk_term.size();
    g.J = up(J);
    g.ldj = ldj;
    g.jabs = up(jabs);
    g.status = up(status);
    ColourGemmArgs c;
    c.J = up(J);  // the first launch's colour amplitudes (set below)
    c.n_pairs = n;
    c.m = P.n_jamp; c.ldj = ldj; c.kp = T.kp; c.np = T.np; c.nc = T.nc;
    c.b_hi = up(T.hi);
    c.b_lo = T.exact ? nullptr : up(T.lo);
    c.inv_den = 1.0 / (double)P.cf_den;
    c.pairval = up(pv);
    c.status = g.status;
    auto launched = [&](cudaError_t e) {  // its status word
      ck(e, "launch");
      ck(cudaDeviceSynchronize(), "kernel");
      int v = 0;
      ck(cudaMemcpy(&v, g.status, sizeof v, cudaMemcpyDeviceToHost), "status");
      ck(cudaMemset(g.status, 0, sizeof v), "status");
      return v;
    };
    // a diagram amplitude's share in colour amplitude alpha, for the reference
    std::vector<std::vector<std::pair<int, double>>> row(P.n_jamp);
    int d = 0;
    for (const Op& op : P.ops) {
      if (!is_amp_op(op.type)) continue;
      for (uint32_t k = 0; k < op.col_count; ++k) {
        const ColEntry& e = P.col[op.col_begin + k];
        row[e.alpha].push_back({M.row[d], amp_negated(op) ? -(double)e.re : (double)e.re});
      }
      ++d;
    }
    std::vector<float> J0;
    std::vector<double> pv0;
    int expired[2] = {0, 0};
    for (uint32_t polls : {kDefault, 0u, kDefault, 1u, 2u, 3u, 4u, 8u, 16u, 64u, 256u, kDefault}) {
      g.spin_limit = c.spin_limit = polls;
      const bool whole = polls == kDefault;
      int v = launched(launch_jamp_gemm(g, sms, nullptr));
      need(whole ? v == 0 : (v == 0 || v == 1), "status of the colour-amplitude GEMM");
      need(polls != 0 || v == 1, "no poll, no expiry (colour amplitudes)");
      expired[0] += v;
      if (whole) {
        ck(cudaMemcpy(J.data(), g.J, J.size() * 4, cudaMemcpyDeviceToHost), "J");
        if (J0.empty()) {
          J0 = J;
          ck(cudaMemcpy(const_cast<float*>(c.J), J0.data(), J0.size() * 4, cudaMemcpyHostToDevice), "J");
          for (int64_t p : {(int64_t)0, (int64_t)63, n / 2, n - 1})
            for (int ri = 0; ri < 2; ++ri)
              for (int a = 0; a < P.n_jamp; ++a) {
                double ref = 0, mag = 0;
                for (auto& x : row[a]) {
                  const double t = x.second * A[(size_t)x.first * lda + 2 * p + ri];
                  ref += t;
                  mag += std::fabs(t);
                }
                // FP32 result, digits cut 27 bits or more below the row's largest amplitude
                need(std::fabs(J0[(size_t)(2 * p + ri) * ldj + a] - ref) <= 2e-7 * mag + 1e-7 * std::fabs(ref), "colour amplitude");
              }
        }
        need(!std::memcmp(J.data(), J0.data(), J.size() * 4), "colour amplitudes after an expiry");
      }
      v = launched(launch_colour_gemm(c, sms, nullptr));
      need(whole ? v == 0 : (v == 0 || v == 1), "status of the colour-sum GEMM");
      need(polls != 0 || v == 1, "no poll, no expiry (colour sum)");
      expired[1] += v;
      if (whole) {
        ck(cudaMemcpy(pv.data(), c.pairval, n * 8, cudaMemcpyDeviceToHost), "pairval");
        if (pv0.empty()) pv0 = pv;
        need(!std::memcmp(pv.data(), pv0.data(), n * 8), "colour sum after an expiry");
      }
    }
    std::printf("%s %d %d\n", argv[arg], expired[0], expired[1]);
    for (const void* q : {(const void*)g.A, (const void*)g.rowmax, (const void*)g.tiles, (const void*)g.chunks, (const void*)g.split_begin,
                          (const void*)g.kk_index, (const void*)g.kk_term, (const void*)g.J, (const void*)g.jabs, (const void*)c.J,
                          (const void*)c.b_hi, (const void*)c.b_lo, (const void*)c.pairval, (const void*)g.status})
      cudaFree(const_cast<void*>(q));
  }
  return faults ? 1 : 0;
}
