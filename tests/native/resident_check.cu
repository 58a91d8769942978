// Residency of the straight-line kernels as planned (amp_kernel.cu, gen_resident)
// against the runtime's occupancy query in a process that has launched nothing, for
// every emitted kernel and tile that can be planned.  Exit status 1 on a difference.
#include <cuda_runtime.h>

#include <cstdio>
#include <vector>

#include "kernels.h"

int main() {
  int bad = 0, n = 0, sm = 0;
  if (cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, 0) != cudaSuccess) return 2;
  const std::vector<std::vector<int>> procs = {{21, 21, 21, 21}, {2, -2, 21, 21}, {2, 2, 2, 2}, {21, 21, 21, 21, 21},
                                               {2, -2, 21, 21, 21}, {2, 2, 2, 2, 21}};
  for (const auto& pdg : procs) {
    const mea::GenEntry* g = mea::find_generated(pdg.data(), (int)pdg.size());
    if (!g) return 3;
    for (int rv = 0; rv < 7; ++rv) {
      const void* k = g->kernel(rv == 6, rv % 6);
      cudaFuncAttributes fa;
      if (cudaFuncGetAttributes(&fa, k) != cudaSuccess) return 4;
      for (int threads = 32; threads <= fa.maxThreadsPerBlock && threads <= 256; threads += 32)
        for (size_t smem = 528; smem <= (48u << 10) - (size_t)fa.sharedSizeBytes; smem += 1204) {
          int want = 0;
          if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&want, k, threads, smem) != cudaSuccess) return 5;
          const int got = mea::gen_resident(fa.numRegs, threads, smem, (size_t)sm);
          ++n;
          if (got != want && ++bad <= 20)
            std::printf("%d registers, %d threads, %zu bytes: %d, the runtime says %d\n", fa.numRegs, threads, smem, got, want);
        }
    }
  }
  std::printf("%d tiles, %d differences\n", n, bad);
  return bad ? 1 : 0;
}
