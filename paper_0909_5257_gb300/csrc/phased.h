// Phased layout of a process program: the tensor-core path's amplitude stage
// with every wavefunction in shared memory (amp_phased_kernel.cu).
//
// A CTA evaluates one event.  Every wavefunction the program stores is
// evaluated once per helicity pattern of its own legs (variant; helshare.h has
// the numbering) into a shared-memory area of 32-byte variants; the currents
// of n_ext - 2 legs, each read by one diagram amplitude only, never leave the
// registers of the lane that makes them (fused units).  The program is cut
// into phases with one CTA barrier after each: the stored values level by
// level (level k: k legs), then, where the values of n_ext - 3 legs do not all
// fit beside each other, one phase per block of their leg sets: no unit reads
// two of them, so the units of a leg set run while its values sit in one of
// two block buffers and the next block's values are made into the other.
// A phase is a list of units, each run by one warp:
//   PRODUCE  32 (op, variant) items of one op type at a time;
//   OUTER    diagram amplitudes = free wavefunctions (up to kPhFree) x up to
//            four vertex partials over complementary leg sets, a lane per
//            helicity combination, the partials held in registers;
//   FUSED    currents of n_ext - 2 legs, a lane per variant, each contracted
//            with the variants of its partial (a round per variant);
//   GENERIC  the remaining diagram amplitudes, a lane per combination.
// The operations and their inputs are the per-lane program's (heget.cuh), so
// the diagram amplitudes are the same bit for bit.
#pragma once
#include <cstdint>
#include <vector>

#include "generator.h"

namespace mea {

enum PhType : uint8_t { PH_PRODUCE = 0, PH_OUTER = 1, PH_FUSED = 2, PH_GENERIC = 3 };
constexpr int kPhFree = 24;     // free wavefunctions per OUTER unit
constexpr int kPhPartials = 4;  // partials per OUTER unit
constexpr int kPhRounds = 4;    // variants of a two-leg partial
constexpr int kPhWarps = 12;    // unit lists per phase; the warps of a CTA divide it

struct PhUnit {
  uint8_t type;   // PhType
  uint8_t op;     // PRODUCE, FUSED: op type; OUTER: 1 plain (spinor) contraction
  uint16_t n;     // items, free wavefunctions, currents, amplitudes
  uint32_t rec;   // first record (16-byte words)
  uint8_t sf, sp;  // OUTER: legs of the free side and of the partials
  uint8_t pass;    // OUTER, GENERIC: combinations 32 pass .. 32 pass + 31
  uint8_t np;      // OUTER: partials
  uint16_t set;    // FUSED: leg-set table
  uint8_t lanes;   // FUSED: log2 of the lanes per current
  uint8_t rounds;  // FUSED: rounds in which some lane has a combination
};
static_assert(sizeof(PhUnit) == 16, "PhUnit must stay 16 bytes");

// PRODUCE item: area offsets (variants) of the output and the inputs, rows of
// the event table, x: EXT leg | helicity bit << 4, PIOV free argument.
struct PhItem {
  uint16_t out, in[3];
  uint8_t r[3], x;
  uint32_t pad;
};
static_assert(sizeof(PhItem) == 16, "PhItem must stay 16 bytes");

// The records of the inner loops hold 32-bit words that are used as they are:
// byte offsets into the area (variants of 32 bytes), into the event table's
// rows (32 bytes each), rows of the amplitude buffer.

// OUTER: one header of four partial blocks, then per free wavefunction its
// block, and per partial the amplitude's row (kPhNone: absent) and weight.
constexpr uint32_t kPhNone = 0xFFFFFFFFu;
struct PhOuterHead {
  uint32_t p[4];
};
struct PhOuterRec {
  uint32_t f, pad[3];
  uint32_t d[4];
  float w[4];
};
static_assert(sizeof(PhOuterHead) == 16 && sizeof(PhOuterRec) == 48, "OUTER records");

// FUSED: per current its input blocks, the inputs' legs (byte offset into
// PhSet::sub), its rows, the partial's block, the amplitude's row and weight.
struct PhFusedRec {
  uint32_t in[3], d;
  uint32_t m[3];
  float w;
  uint32_t r[3], p;
};
static_assert(sizeof(PhFusedRec) == 48, "FUSED record");

struct PhGenericRec {
  uint8_t type, flags;  // flags: ADOT's leg bits
  uint16_t d;
  uint16_t in[4];
  uint8_t m[4];  // legs of the inputs
  uint8_t r[3], pad;
  float w;
  uint32_t pad2[2];
};
static_assert(sizeof(PhGenericRec) == 32, "GENERIC record");

// FUSED: a leg set's variants that occur in the sum and, per round, the
// partial's variant (low byte) and combination (high byte) of each.
constexpr uint16_t kPhNoPair = 0xFFFFu;
struct PhSet {
  uint8_t v[32];                    // variant of lane i
  uint16_t uh[kPhRounds][32];       // kPhNoPair: none
  uint16_t sub[32][32];             // [input legs, as bits of the set's legs][lane]: the input's variant x 32
};

struct PhProgram {
  std::vector<uint32_t> rec;       // records (16-byte words as 4 x uint32)
  std::vector<PhUnit> units;
  std::vector<int> list_end;       // [phases][kPhWarps]: end of each list's units
  int phases = 0;
  std::vector<PhSet> sets;
  std::vector<uint8_t> hv;         // [2^n_ext][128]: variant of the legs for combination h
  int area = 0;                    // variants per event
  int H = 0;
  double cost = 0;                 // estimated warp instructions per event
  double flops = 0;                // of the evaluated operations per event (op_flop_cost)
};

// lanes: the helicity combinations; weight[d]: sum of the colour coefficients' magnitudes of diagram d
// (JampMap::weight), row[d] its row in the amplitude buffer (JampMap::row).  Throws LayoutError when the program does not have
// the structure above or its area exceeds max_area variants.
PhProgram build_phased(const Program& P, const HelLanes& lanes, const std::vector<float>& weight,
                       const std::vector<int>& row, int max_area);

}  // namespace mea
