// The server's estimate of an event's cost (server.cu, request_cost) against the
// device times per event measured on a GB300 for the five-jet processes, mixed and
// FP64: the ratio of any two must be within a factor of 2 of the measured one.
// Exit status 1 on a fault.
#include <cstdio>
#include <vector>

#include "process.h"

int main() {
  struct Case {
    std::vector<int> pdg;
    double us[2];  // mixed, FP64
  };
  const std::vector<Case> cases = {{{21, 21, 21, 21, 21, 21, 21}, {2.677, 21.63}},
                                   {{2, -2, 21, 21, 21, 21, 21}, {0.909, 8.13}},
                                   {{2, 2, 2, 2, 21, 21, 21}, {0.582, 5.71}}};
  std::vector<double> cost, us;
  for (const Case& c : cases) {
    mea_process_t P = nullptr;
    if (mea_create_process_host_only(c.pdg.data(), (int)c.pdg.size(), nullptr, &P) != MEA_OK) return 2;
    for (int k = 0; k < 2; ++k) {
      cost.push_back(mea::request_cost(P, k == 0 ? MEA_PREC_MIXED : MEA_PREC_FP64));
      us.push_back(c.us[k]);
    }
    mea_destroy_process(P);
  }
  int bad = 0;
  for (size_t i = 0; i < cost.size(); ++i)
    for (size_t j = 0; j < cost.size(); ++j) {
      const double f = cost[i] / cost[j] / (us[i] / us[j]);
      if (!(f < 2.0)) {
        ++bad;
        std::printf("%zu against %zu: %.2f times the measured ratio\n", i, j, f);
      }
    }
  return bad ? 1 : 0;
}
