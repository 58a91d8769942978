// Levels of the ordered recursion (ordered.h), for processes of any size: the items
// of a level run in any order.  Every level runs twice on the same state, its items
// forwards and backwards, on random externals: an item that read what the level
// writes would find it in one of the two orders only (unwritten values are NaN), and
// an amplitude that two items of a level add to would be rounded differently or lose
// its start.  All values must be the same bit for bit, none NaN, and every value of
// the area written by one item only.  Prints per process: name, levels, items; exit
// status 1 on a fault.
#define MEA_HD inline
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "ordered_eval.cuh"

using namespace mea;

static int faults = 0;
static void fault(const char* name, const char* what) {
  if (++faults <= 20) std::printf("%s: %s\n", name, what);
}

int main(int argc, char** argv) {
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
    const OrdProgram Q = build_ordered(P);
    const int n = P.n_ext;
    std::mt19937_64 rng(0x5eed + arg);
    auto u = [&]() { return std::uniform_real_distribution<double>(0.1, 1.0)(rng); };
    std::vector<double> et(8 * n), mt(5 * P.masks.size());
    for (double& x : et) x = u();
    for (double& x : mt) x = u();
    std::vector<int8_t> leg(4 * n, 0);
    for (int l = 0; l < n; ++l) {
      leg[4 * l] = (int8_t)P.leg_type[l];
      leg[4 * l + 2] = (int8_t)P.incoming[l];
    }
    const double nan = std::nan("");
    std::vector<double> area(Q.area, nan), F(2 * (size_t)Q.n_f, nan);
    long long items = 0;
    int levels = 0;
    for (size_t i = 0; i < Q.stages.size(); ++levels) {
      size_t j = i;
      while (j < Q.stages.size() && Q.level[j] == Q.level[i]) ++j;
      struct Item {
        size_t stage;
        int word;
        uint32_t var;
      };
      std::vector<Item> level;
      for (size_t q = i; q < j; ++q)
        for (int w = 0; w < Q.stages[q].words; ++w)
          for (uint32_t v = 0; v < (1u << Q.stages[q].nb); ++v) level.push_back({q, w, v});
      items += (long long)level.size();
      std::vector<double> out[2] = {area, area}, amp[2] = {F, F};
      for (int pass = 0; pass < 2; ++pass)
        for (size_t k = 0; k < level.size(); ++k) {
          const Item& it = level[pass ? level.size() - 1 - k : k];
          const OrdStage& st = Q.stages[it.stage];
          OrdEvent E{out[pass].data(), amp[pass].data(), et.data(), mt.data(), leg.data()};
          ord_item(st, Q.rec.data() + st.rec + (size_t)it.word * st.stride, it.var, E);
        }
      if (std::memcmp(out[0].data(), out[1].data(), out[0].size() * 8)) fault(argv[arg], "a level reads what it writes, or writes twice");
      if (std::memcmp(amp[0].data(), amp[1].data(), amp[0].size() * 8)) fault(argv[arg], "items of a level share an amplitude");
      for (size_t k = 0; k < area.size(); ++k)
        if (area[k] == area[k] && std::memcmp(&area[k], &out[0][k], 8)) { fault(argv[arg], "a value written in two levels"); break; }
      area = out[0];
      F = amp[0];
      i = j;
    }
    for (double x : area)
      if (!(x == x)) { fault(argv[arg], "a value of the area that is NaN or never written"); break; }
    for (double x : F)
      if (!(x == x)) { fault(argv[arg], "an amplitude that is NaN or never written"); break; }
    std::printf("%s %d %lld\n", argv[arg], levels, items);
  }
  return faults ? 1 : 0;
}
