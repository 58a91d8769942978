// Colour amplitudes that are signed sums of others.
#pragma once
#include <cstdint>
#include <vector>

#include "generator.h"

namespace mea {

// J_alpha = sum_d c_{alpha d} A_d: a base of the rows of the coefficients c
// (the first mb colour amplitudes) and the others as sums of it with
// coefficients 1 and -1, exact for every diagram (the Kleiss-Kuijf relations of
// the gluon processes: (n-2)! of the (n-1)!/2 orderings).  mb = n_jamp and empty
// tables where there are none or the base is no prefix.  A handle finds it once (25 ms
// of host time for gg>5g) and hands it to what needs it.
struct ColourBase {
  int mb = 0;
  std::vector<uint16_t> index;  // [3 (n_jamp - mb)]: begin, first subtracted, end in term
  std::vector<uint16_t> term;   // base columns
};
ColourBase find_colour_base(const Program& p);

}  // namespace mea
