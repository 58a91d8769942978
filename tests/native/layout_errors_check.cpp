// Layouts that a process does not have are refused with LayoutError, the one
// exception that a handle takes for a reason to fall back: phased evaluation outside
// 6 and 7 legs, in too small an area, without weights; the recursion without one of
// its momenta.  Exit status 1 on a fault.
#include <cstdio>
#include <stdexcept>

#include "generator.h"
#include "ordered.h"
#include "phased.h"

using namespace mea;

template <class F>
static int refused(F f, const char* what) {
  try {
    f();
  } catch (const LayoutError&) {
    return 0;
  } catch (const std::exception&) {
  }
  std::printf("%s: no LayoutError\n", what);
  return 1;
}

int main() {
  int bad = 0;
  for (int n : {5, 6}) {
    const Program P = build_program(std::vector<int>(n, 21));
    const HelLanes L = helicity_lanes(P);
    const std::vector<float> w(P.n_diagrams, 1.f);
    std::vector<int> row(P.n_diagrams);
    for (int d = 0; d < P.n_diagrams; ++d) row[d] = d;
    bad += refused([&] { build_phased(P, L, w, row, n == 5 ? 6800 : 10); }, n == 5 ? "five legs" : "area");
    if (n == 6) bad += refused([&] { build_phased(P, L, {}, row, 6800); }, "weights");
  }
  Program P = build_program({21, 21, 21, 21, 21});
  P.masks.resize(3);  // a momentum is missing
  bad += refused([&] { build_ordered(P); }, "event table");
  return bad ? 1 : 0;
}
