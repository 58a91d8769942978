// FP64 straight-line body (codegen.cpp) compiled for the host: every colour amplitude
// must be the plain sum of its diagram amplitudes in program order, bit for bit,
// with no colour amplitude formed from others.  BODY_FILE, BODY: the emitted struct;
// argument: the process.  Exit status 1 on a difference.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <numeric>
#include <random>
#include <string>
#include <type_traits>
#include <vector>

#define MEA_HD inline
#define __device__
#define __forceinline__ inline
#include "generator.h"
#include "heget.cuh"

// what gen_kernel.cuh gives the FP64 body; jfin reads the sums off
template <typename R, bool PACKED>
struct JSum {
  cx<R> hi{R(0), R(0)};
};
static std::vector<cx<double>> sums;
template <bool PACKED>
void jadd(JSum<double, PACKED>& J, cx<double> a) { J.hi = J.hi + a; }
template <typename R>
inline cx<R> neg(cx<R> a) { return -a; }
template <bool PACKED>
cx<double> jfin(const JSum<double, PACKED>& J) {
  sums.push_back(J.hi);
  return J.hi;
}
// FP32 only (a body may name them where FP64 does not go)
template <typename T, bool PACKED>
void jadd(JSum<T, PACKED>&, const JSum<T, PACKED>&);
template <typename T, bool PACKED>
void jsub(JSum<T, PACKED>&, const JSum<T, PACKED>&);
#include BODY_FILE

using namespace mea;

int main(int, char** argv) {
  std::vector<int> pdg;
  std::string s = argv[1];
  for (size_t p = 0; p < s.size();) {
    size_t e = s.find(',', p);
    if (e == std::string::npos) e = s.size();
    pdg.push_back(std::atoi(s.substr(p, e - p).c_str()));
    p = e + 1;
  }
  BuildOptions order;
  order.group_together = true;  // the order the bodies are emitted in
  const Program P = build_program(pdg, order);
  const int n = P.n_ext, m = P.n_jamp;
  int f = 0;
  for (const ColEntry& c : P.col) f = std::gcd(f, std::abs((int)c.re));
  if (f <= 0 || (f & (f - 1)) != 0) f = 1;
  std::mt19937_64 rng(0x5eed);
  auto u = [&]() { return std::uniform_real_distribution<double>(-1, 1)(rng); };
  const double g = 1.2;
  int bad = 0;
  for (int trial = 0; trial < 50; ++trial) {
    std::vector<double> et(8 * n), mt(5 * P.masks.size());
    for (double& x : et) x = u();
    for (double& x : mt) x = u();
    const uint32_t lam = (uint32_t)rng() & ((1u << n) - 1u);
    double val = 0;
    float kappa = 0;
    sums.clear();
    BODY<double>::run(et.data(), mt.data(), lam, g, g * g, 1.0, val, kappa);
    std::vector<W4<double>> slots(P.n_slots);
    std::vector<cx<double>> J(m, cx<double>{0, 0});
    const double* M = mt.data();
    for (const Op& op : P.ops) {
      W4<double> x[4], w{};
      cx<double> a{0, 0};
      const int n_in = op.type == OP_EXT ? 0 : op.n_in;
      for (int k = 0; k < n_in; ++k) x[k] = slots[op.in[k]];
      const double *k0 = M + 5 * op.min[0], *k1 = M + 5 * op.min[1], *k2 = M + 5 * op.min[2], *q = M + 5 * op.mout;
      switch (op.type) {
        case OP_EXT: {
          const double* o = &et[8 * op.leg];
          const int h = (lam >> op.leg & 1u) ? 1 : -1, in = P.incoming[op.leg];
          const int kind = P.leg_type[op.leg] == 1 ? (in ? 0 : 1) : (in ? 3 : 2);
          w = P.leg_type[op.leg] == 0 ? ext_gluon<double>(o, o + 3, h, !in)
                                      : ext_spinor<double>(o[0], o[1], mk<double>(o[2], o[3]), h, kind);
          break;
        }
        case OP_JVV: w = jvv<double>(x[0], x[1], k0, k1, q[4], g); break;
        case OP_JGGG: w = jggg<double>(x[0], x[1], x[2], q[4], g * g); break;
        case OP_FVI: w = fvi<double>(x[0], x[1], q, q[4], g); break;
        case OP_FVO: w = fvo<double>(x[0], x[1], q, q[4], g); break;
        case OP_JIO: w = jio<double>(x[0], x[1], q[4], g); break;
        case OP_PVVV: w = vvv_part<double>(x[0], x[1], k0, k1, k2, g); break;
        case OP_PGGGG: w = gggg_part<double>(x[0], x[1], x[2], g * g); break;
        case OP_PIOV: w = op.leg == 0 ? iov_part_i<double>(x[0], x[1], g) : op.leg == 1 ? iov_part_o<double>(x[0], x[1], g) : iov_part_v<double>(x[0], x[1], g); break;
        case OP_AVVV: a = vvv_amp<double>(x[0], x[1], x[2], k0, k1, k2, g); break;
        case OP_AGGGG: a = gggg_amp<double>(x[0], x[1], x[2], x[3], g * g); break;
        case OP_AIOV: a = iov_amp<double>(x[0], x[1], x[2], g); break;
        case OP_ADOT: a = part_contract<double>(x[0], x[1], op.leg & 1, op.leg & 2); break;
      }
      if (!is_amp_op(op.type)) { slots[op.out] = w; continue; }
      for (uint32_t k = 0; k < op.col_count; ++k) {
        const ColEntry& c = P.col[op.col_begin + k];
        J[c.alpha] = J[c.alpha] + (double)(c.re / f) * a;
      }
    }
    if ((int)sums.size() != m) ++bad;
    for (int a = 0; a < m && (int)sums.size() == m; ++a)
      if (sums[a].r != J[a].r || sums[a].i != J[a].i) ++bad;
  }
  std::printf("%s: %d colour amplitudes, %d differences\n", argv[1], m, bad);
  return bad ? 1 : 0;
}
