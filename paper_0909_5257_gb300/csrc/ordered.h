// Ordered-recursion layout of a process: the FP64 path's |M|^2 through
// colour-ordered off-shell currents (Berends and Giele 1988) instead of one
// amplitude per Feynman diagram.
//
// The FP64 pipe of this GPU runs at 1/64 of the FP32 pipe, so on the FP64 path
// only the number of FP64 operations counts.  The sum of all diagrams of one
// colour ordering obeys a recursion over ordered words of legs,
//   P^2 J(w) = sum_{w=uv} [J(u), J(v)] + sum_{w=uvt} {J(u), J(v), J(t)}
//   [a, b] = ((2 Pb + Pa).a) b - ((2 Pa + Pb).b) a + (Pa - Pb) (a.b)
//   {a, b, c} = 2 (a.c) b - (a.b) c - (b.c) a
// (momenta flowing out; the three- and four-gluon Feynman rules with their
// colour factors expanded in products of generators), quark words
//   P^2 psi(w) = Pslash sum_{w=uv} Jslash(u) psi(v),
//   P^2 psibar(w) = -(sum_{w=vu} psibar(v) Jslash(u)) Pslash,
// and, with two quark lines, a composite letter x(t, u): the gluon current
// psibar(t) gamma psi(u) / P^2 of the second line, which enters the words of the
// first line as an off-shell gluon.  Every word current is evaluated once per
// helicity pattern of its letters.  A quark line of one chirality needs two of
// a spinor's four components; |M_h|^2 is the same for a helicity combination
// and its flipped one (parity), so one of each pair is evaluated: the first
// quark line right-handed, or leg 0 of a pure-gluon process with helicity -1.
//
// Colour amplitudes: the base of the ordered traces (ColourBase, pure gluons: the
// words that start with leg 0), the strings of one quark line, or the pairs of
// strings of two lines, contracted with the integer colour matrix as before.
//
// A program is a list of stages by level, with one CTA barrier after each level
// (the stages of a level read nothing that it writes); a stage is a list of words
// of one form (same number of letters and of helicity bits), an item one word and
// one helicity pattern.  Patterns are numbered by the letters' bits in word order,
// the first letter highest.  Currents of as many letters as a colour ordering less
// one (fused) are not stored: their items close them with the remaining letter at
// once.
#pragma once
#include <cstdint>
#include <vector>

#include "colour_base.h"
#include "generator.h"

#ifndef MEA_HD
#define MEA_HD __host__ __device__ __forceinline__
#endif

namespace mea {

enum OrdType : uint8_t {
  ORD_EXT_G = 0,    // polarisation vector of a gluon letter
  ORD_EXT_Q = 1,    // column or row two-spinor of a quark leg
  ORD_G = 2,        // gluon word
  ORD_GF = 3,       // gluon word closed at once (fused)
  ORD_GA = 4,       // pure-gluon ordering: its vertices at the root, closed with both root polarisations
  ORD_PSI = 5,      // quark word
  ORD_BAR = 6,      // barred quark word
  ORD_PF = 7,       // quark word closed at once with a gluon letter and the row
  ORD_X = 8,        // gluon current of a quark line
  ORD_Z = 9,        // [J(x), eps_root] of a letter x for both root polarisations
  ORD_PA = 10,      // quark line's ordering: row . sum Jslash(u) psi(v)
};

struct OrdStage {
  uint8_t type;
  uint8_t k;      // letters
  uint8_t nb;     // helicity bits of an item
  uint8_t full;   // gluon words with a composite letter: currents that are not conserved
  uint16_t words;
  uint16_t stride;  // words of 8 bytes per record
  uint32_t rec;   // first record (8-byte words)
};
static_assert(sizeof(OrdStage) == 12, "OrdStage");

// Reference to a stored current: area offset (16-byte units), event-table row
// of its legs, where its bits lie in the item's pattern.
struct OrdRef {
  uint16_t off;
  uint8_t row;
  uint8_t sh, nb;
  uint8_t flags;  // 1: stored word reversed (bits reversed), 2: negated
  uint16_t pad;
};
static_assert(sizeof(OrdRef) == 8, "OrdRef");

// Closing of a fused current: colour ordering's first amplitude (F index), the
// closing value (area offset; for pure gluons [x bits][root bit]), the bits of x, whether x
// stands left of the word, whether the word enters reversed, its sign.
struct OrdClose {
  uint16_t f, z;
  uint8_t xnb, left, rev, neg;
};
static_assert(sizeof(OrdClose) == 8, "OrdClose");

struct OrdProgram {
  std::vector<OrdStage> stages;
  std::vector<int> level;          // of every stage: a barrier stands where it grows
  std::vector<uint64_t> rec;
  std::vector<uint16_t> fidx;      // [n_colour][H]: F index of ordering a for evaluated combination h
  std::vector<int> range;          // [H][2]: orderings that contribute to combination h
  std::vector<double> kmat;        // [n_colour][n_colour] colour matrix of the orderings
  int n_colour = 0, H = 0;
  int area = 0;                    // doubles per event
  int n_f = 0;                     // amplitudes (complex) per event
  double norm = 0;                 // |M|^2 = norm g^(2n-4) sum_h J K J^*, parity and averages included
};

// Throws LayoutError when a word needs a momentum the program's event
// table does not hold or a table does not fit its type.
// base: find_colour_base(P), found here when null
OrdProgram build_ordered(const Program& P, const ColourBase* base = nullptr);

}  // namespace mea
