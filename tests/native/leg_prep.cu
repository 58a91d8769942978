// FP64 leg preparation of gluons (amp_common.cuh): the polarisation basis of
// momenta with integer components, whose squares and their sums are exact, must be
// the correctly rounded roots and quotients that the host's FP64 arithmetic gives,
// bit for bit.  Prints the number of momenta; exit status 1 on a difference.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <type_traits>
#include <vector>

#include "../../include/mea.h"
#include "amp_common.cuh"

using namespace mea;

__global__ void prep_kernel(const DevProgram P, const double* mom, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) prep_leg<double>(P, mom + 4 * (size_t)i, 0, out + 8 * (size_t)i);
}

static void ck(cudaError_t e) {
  if (e == cudaSuccess) return;
  std::printf("%s\n", cudaGetErrorString(e));
  std::exit(2);
}

int main() {
  std::vector<double> mom;
  std::mt19937_64 rng(0x5eed);
  auto add = [&](double x, double y, double z) {
    for (double v : {std::sqrt(x * x + y * y + z * z), x, y, z}) mom.push_back(v);
  };
  for (int k = 0; k < 20000; ++k) {  // 3 to 24 bits a component: sums of squares below 2^50
    const int b = 3 + k % 22;
    auto u = [&]() { return (double)((int64_t)(rng() % (2ull << b)) - (int64_t)(1ull << b)); };
    add(u(), u(), u());
  }
  add(0, 0, 7); add(0, 0, -7); add(3, 0, 0); add(0, -3, 0); add(-3, 4, 0); add(1, 0, 16777215); add(0, 1, -16777215);
  const int n = (int)(mom.size() / 4);
  std::vector<double> got(8 * (size_t)n);
  const int8_t leg[4] = {0, 0, 0, 0};
  void *dm, *dl, *dr;
  ck(cudaMalloc(&dm, mom.size() * 8));
  ck(cudaMalloc(&dr, got.size() * 8));
  ck(cudaMalloc(&dl, sizeof leg));
  ck(cudaMemcpy(dm, mom.data(), mom.size() * 8, cudaMemcpyHostToDevice));
  ck(cudaMemcpy(dl, leg, sizeof leg, cudaMemcpyHostToDevice));
  DevProgram P;
  P.n_ext = 1;
  P.leg_info = static_cast<const int8_t*>(dl);
  prep_kernel<<<(n + 127) / 128, 128>>>(P, static_cast<const double*>(dm), static_cast<double*>(dr), n);
  ck(cudaGetLastError());
  ck(cudaMemcpy(got.data(), dr, got.size() * 8, cudaMemcpyDeviceToHost));
  int bad = 0;
  for (int i = 0; i < n; ++i) {
    const double x = mom[4 * i + 1], y = mom[4 * i + 2], z = mom[4 * i + 3];
    const double kt = std::sqrt(x * x + y * y), kk = std::sqrt(x * x + y * y + z * z);
    double ct = z < 0 ? -1 : 1, st = 0, cp = 1, sp = 0;
    if (kt > 0) { ct = z / kk; st = kt / kk; cp = x / kt; sp = y / kt; }
    const double want[6] = {ct * cp, ct * sp, -st, -sp, cp, 0.0};
    for (int k = 0; k < 6; ++k)
      if (got[8 * (size_t)i + k] != want[k] && ++bad <= 10)
        std::printf("(%g, %g, %g) component %d: %.17g, not %.17g\n", x, y, z, k, got[8 * (size_t)i + k], want[k]);
  }
  std::printf("%d momenta, %d differences\n", n, bad);
  return bad ? 1 : 0;
}
