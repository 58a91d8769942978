// Host check of the phased layout (phased.h): for every process given on the
// command line the units are run phase by phase in FP64, lane by lane as
// amp_phased_kernel.cu runs them, with the vertex functions of heget.cuh, and
// every diagram amplitude of every summed helicity combination must equal the
// per-lane program's bit for bit and be written exactly once.  Within a phase
// nothing may be read that the phase writes or that no earlier phase wrote,
// and every offset must lie inside the area.  Prints per process: name,
// amplitudes compared, mismatches, area; exit status 1 on any fault.
#define MEA_HD inline
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <set>
#include <string>
#include <vector>

#include "generator.h"
#include "heget.cuh"
#include "phased.h"

using namespace mea;
typedef W4<double> V;

static int faults = 0;
static void fault(const char* what) {
  if (++faults <= 20) std::printf("fault: %s\n", what);
}
static const double g = 1.1, gg = g * g;

struct Inputs {
  std::vector<std::vector<V>> ext;  // [leg][lambda bit]
  std::vector<double> mt;
};

static V made(int type, int leg, const V* x, const double* k0, const double* k1, const double* k2, const double* q) {
  switch (type) {
    case OP_JVV: return jvv<double>(x[0], x[1], k0, k1, q[4], g);
    case OP_JGGG: return jggg<double>(x[0], x[1], x[2], q[4], gg);
    case OP_FVI: return fvi<double>(x[0], x[1], q, q[4], g);
    case OP_FVO: return fvo<double>(x[0], x[1], q, q[4], g);
    case OP_JIO: return jio<double>(x[0], x[1], q[4], g);
    case OP_PVVV: return vvv_part<double>(x[0], x[1], k0, k1, k2, g);
    case OP_PGGGG: return gggg_part<double>(x[0], x[1], x[2], gg);
    case OP_PIOV:
      return leg == 0 ? iov_part_i<double>(x[0], x[1], g) : (leg == 1 ? iov_part_o<double>(x[0], x[1], g) : iov_part_v<double>(x[0], x[1], g));
  }
  fault("unknown op");
  return x[0];
}
static cx<double> closed(int type, int flags, const V* x, const double* k0, const double* k1, const double* k2) {
  switch (type) {
    case OP_AVVV: return vvv_amp<double>(x[0], x[1], x[2], k0, k1, k2, g);
    case OP_AGGGG: return gggg_amp<double>(x[0], x[1], x[2], x[3], gg);
    case OP_AIOV: return iov_amp<double>(x[0], x[1], x[2], g);
  }
  return part_contract<double>(x[0], x[1], (flags & 1) != 0, (flags & 2) != 0);
}

int main(int argc, char** argv) {
  for (int a = 1; a < argc; ++a) {
    std::vector<int> pdg;
    std::string s = argv[a];
    for (size_t p = 0; p < s.size();) {
      size_t e = s.find(',', p);
      if (e == std::string::npos) e = s.size();
      pdg.push_back(std::atoi(s.substr(p, e - p).c_str()));
      p = e + 1;
    }
    const Program P = build_program(pdg);
    const HelLanes lanes = helicity_lanes(P);
    const int n = P.n_ext, H = lanes.n;
    std::vector<float> weight(P.n_diagrams);
    for (int d = 0; d < P.n_diagrams; ++d) weight[d] = 1.f + (float)(d % 7);
    std::vector<int> row_of(P.n_diagrams), row(P.n_diagrams);  // a permutation
    for (int d = 0; d < P.n_diagrams; ++d) row[d] = (int)((d * 5LL + 3) % P.n_diagrams);
    if (P.n_diagrams % 5 == 0)
      for (int d = 0; d < P.n_diagrams; ++d) row[d] = P.n_diagrams - 1 - d;
    for (int d = 0; d < P.n_diagrams; ++d) row_of[row[d]] = d;
    std::vector<char> negated;
    for (const Op& op : P.ops)
      if (is_amp_op(op.type)) negated.push_back(amp_negated(op));
    const PhProgram Q = build_phased(P, lanes, weight, row, 6800);

    std::mt19937_64 rng(0x5eed + a);
    auto u = [&]() { return std::uniform_real_distribution<double>(-1.0, 1.0)(rng); };
    Inputs in;
    in.ext.assign(n, std::vector<V>(2));
    for (auto& l : in.ext)
      for (auto& w : l)
        for (int k = 0; k < 4; ++k) w.c[k] = {u(), u()};
    std::vector<double> leg(4 * n);
    for (double& x : leg) x = u();
    in.mt.assign(5 * P.masks.size(), 0.0);
    for (size_t r = 0; r < P.masks.size(); ++r) {
      double* q = &in.mt[5 * r];
      for (int l = 0; l < n; ++l)
        if (P.masks[r] >> l & 1u)
          for (int m = 0; m < 4; ++m) q[m] += leg[4 * l + m];
      q[4] = 1.0 / (q[0] * q[0] - q[1] * q[1] - q[2] * q[2] - q[3] * q[3]);
    }
    auto mrow = [&](int r) -> const double* {
      if (5 * (size_t)r + 5 > in.mt.size()) { fault("event-table row"); return in.mt.data(); }
      return &in.mt[5 * (size_t)r];
    };

    // per combination through the slots
    std::vector<cx<double>> ref((size_t)H * P.n_diagrams), got(ref.size());
    std::vector<int> written(ref.size(), 0);
    for (int h = 0; h < H; ++h) {
      std::vector<V> slots(P.n_slots);
      int d = 0;
      for (const Op& op : P.ops) {
        V x[4];
        const int n_in = op.type == OP_EXT ? 0 : op.n_in;
        for (int k = 0; k < n_in; ++k) x[k] = slots[op.in[k]];
        if (is_amp_op(op.type))
          ref[(size_t)h * P.n_diagrams + d++] = closed(op.type, op.leg, x, mrow(op.min[0]), mrow(op.min[1]), mrow(op.min[2]));
        else if (op.type == OP_EXT)
          slots[op.out] = in.ext[op.leg][lanes.hel[(size_t)h * n + op.leg] > 0];
        else
          slots[op.out] = made(op.type, op.leg, x, mrow(op.min[0]), mrow(op.min[1]), mrow(op.min[2]), mrow(op.mout));
      }
    }

    std::vector<V> area(Q.area);
    std::vector<char> have(Q.area, 0);
    size_t i = 0;
    for (int ph = 0; ph < Q.phases; ++ph) {
      std::set<int> rd, wr;
      auto ld = [&](uint32_t k) -> V {
        if (k >= (uint32_t)Q.area || !have[k]) { fault("read outside the area or before it is written"); return area[0]; }
        rd.insert((int)k);
        return area[k];
      };
      std::vector<std::pair<int, V>> made_here;
      auto take = [&](cx<double> z, uint32_t d, float w, uint32_t h) {
        if (d >= (uint32_t)P.n_diagrams) { fault("row"); return; }
        const uint32_t dd = (uint32_t)row_of[d];
        if (dd >= (uint32_t)P.n_diagrams || h >= (uint32_t)H) { fault("diagram or combination"); return; }
        if (w != weight[dd]) fault("weight");
        if (negated[dd]) z = -z;  // the sign the coefficients carry
        got[(size_t)h * P.n_diagrams + dd] = z;
        ++written[(size_t)h * P.n_diagrams + dd];
      };
      for (; i < (size_t)Q.list_end[ph * kPhWarps + kPhWarps - 1]; ++i) {
        const PhUnit& U = Q.units[i];
        auto rec = [&](size_t at, void* to, size_t bytes) {
          if (4 * (U.rec + at) + bytes / 4 > Q.rec.size()) { fault("record"); std::memset(to, 0, bytes); return; }
          std::memcpy(to, &Q.rec[4 * (U.rec + at)], bytes);
        };
        for (int lane = 0; lane < 32; ++lane) {
          if (U.type == PH_PRODUCE) {
            for (int k = lane; k < U.n; k += 32) {
              PhItem it;
              rec(k, &it, sizeof it);
              V x[4], y;
              const int n_in = U.op == OP_EXT ? 0 : (U.op == OP_JGGG || U.op == OP_PGGGG ? 3 : 2);
              for (int j = 0; j < n_in; ++j) x[j] = ld(it.in[j]);
              if (U.op == OP_EXT) y = in.ext.at(it.x & 15)[it.x >> 4];
              else y = made(U.op, it.x, x, mrow(it.r[0]), mrow(it.r[1]), mrow(it.r[2]), mrow(it.r[2]));
              if (it.out >= Q.area) fault("output outside the area");
              else made_here.push_back({it.out, y});
            }
          } else if (U.type == PH_FUSED) {
            if (U.set >= Q.sets.size()) { fault("set"); continue; }
            const PhSet& T = Q.sets[U.set];
            const int per = 32 >> U.lanes;
            for (int t = lane >> U.lanes; t < U.n; t += per) {
              PhFusedRec c;
              rec(3 * t, &c, sizeof c);
              V x[4];
              for (int j = 0; j < (U.op == OP_JGGG ? 3 : 2); ++j) x[j] = ld((c.in[j] + T.sub[c.m[j] / 64][lane]) / 32);
              const V y = made(U.op, 0, x, mrow(c.r[0] / 32), mrow(c.r[1] / 32), mrow(c.r[2] / 32), mrow(c.r[2] / 32));
              for (int r = 0; r < kPhRounds; ++r)
                if (T.uh[r][lane] != kPhNoPair)
                  take(part_contract<double>(y, ld(c.p / 32 + (T.uh[r][lane] & 255)), U.op == OP_FVI || U.op == OP_FVO, false), c.d, c.w,
                       T.uh[r][lane] >> 8);
            }
          } else {
            const int h = 32 * U.pass + lane;
            if (h >= H) continue;
            if (U.type == PH_OUTER) {
              PhOuterHead hd;
              rec(0, &hd, sizeof hd);
              for (int k = 0; k < U.n; ++k) {
                PhOuterRec c;
                rec(1 + 3 * k, &c, sizeof c);
                for (int q = 0; q < U.np; ++q)
                  take(part_contract<double>(ld(c.f / 32 + Q.hv[128 * U.sf + h]), ld(hd.p[q] / 32 + Q.hv[128 * U.sp + h]), U.op != 0, false),
                       c.d[q], c.w[q], h);
              }
            } else {
              for (int k = 0; k < U.n; ++k) {
                PhGenericRec c;
                rec(2 * k, &c, sizeof c);
                V x[4];
                const int n_in = c.type == OP_AGGGG ? 4 : (c.type == OP_ADOT ? 2 : 3);
                for (int j = 0; j < n_in; ++j) x[j] = ld(c.in[j] + Q.hv[128 * c.m[j] + h]);
                take(closed(c.type, c.flags & 1, x, mrow(c.r[0]), mrow(c.r[1]), mrow(c.r[2])), c.d, c.w, h);
              }
            }
          }
        }
      }
      for (auto& m : made_here) {
        if (rd.count(m.first)) fault("written in the phase that reads it");
        if (!wr.insert(m.first).second) fault("written twice in a phase");
        area[m.first] = m.second;
        have[m.first] = 1;
      }
    }
    if (i != Q.units.size()) fault("units beyond the last phase");
    int64_t bad = 0;
    for (size_t k = 0; k < ref.size(); ++k)
      if (written[k] != 1 || std::memcmp(&ref[k], &got[k], sizeof ref[k]) != 0) ++bad;
    if (bad) ++faults;
    std::printf("%s %zu %lld %d\n", argv[a], ref.size(), (long long)bad, Q.area);
  }
  return faults ? 1 : 0;
}
