// Bounded waits of the tensor-core GEMMs that run out: a wait with the usual
// limit that nothing ends takes seconds.  Prints its time; exit status 1 on a fault.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <vector>

#include "colour_gemm.h"
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

int main() {
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
  return faults ? 1 : 0;
}
