// Phased layout of a process program (see phased.h).
#include "phased.h"

#include <algorithm>
#include <cstring>
#include <map>
#include <stdexcept>
#include <string>

namespace mea {
namespace {

// All stored values stay beside each other up to this many variants (32 KB):
// three to six CTAs per SM still fit, and no block phases are needed.
constexpr int kResidentArea = 1024;
// Variants of one block buffer: leg sets are merged into a block up to here
// (fewer barriers), a larger set is a block of its own.
constexpr int kBlockArea = 768;

uint32_t pext8(uint32_t x, uint32_t S) {
  uint32_t r = 0;
  int k = 0;
  for (int l = 0; l < 8; ++l)
    if (S >> l & 1u) {
      if (x >> l & 1u) r |= 1u << k;
      ++k;
    }
  return r;
}
uint32_t pdep8(uint32_t v, uint32_t S) {
  uint32_t r = 0;
  int k = 0;
  for (int l = 0; l < 8; ++l)
    if (S >> l & 1u) {
      if (v >> k & 1u) r |= 1u << l;
      ++k;
    }
  return r;
}

struct Costed {
  PhUnit u;
  double cost;
  int phase;  // -1: any consuming phase
};

void check(bool ok, const char* why) {
  if (!ok) throw LayoutError(std::string("phased layout: ") + why);
}

}  // namespace

PhProgram build_phased(const Program& P, const HelLanes& lanes, const std::vector<float>& weight,
                       const std::vector<int>& row, int max_area) {
  const int n = P.n_ext, H = lanes.n;
  check(n >= 6 && n <= 7, "6 or 7 legs");
  check(H >= 1 && H <= 128, "at most 128 combinations");
  check(P.masks.size() <= 256, "at most 256 event-table rows");
  const int n_ops = (int)P.ops.size();
  const uint32_t all = (1u << n) - 1u;
  PhProgram Q;
  Q.H = H;

  std::vector<uint32_t> hbits(H, 0);
  for (int h = 0; h < H; ++h)
    for (int l = 0; l < n; ++l)
      if (lanes.hel[(size_t)h * n + l] > 0) hbits[h] |= 1u << l;
  Q.hv.assign((size_t)128 << n, 0);
  for (uint32_t S = 0; S <= all; ++S)
    for (int h = 0; h < H; ++h) Q.hv[S * 128 + h] = (uint8_t)pext8(hbits[h], S);
  auto used = [&](uint32_t S) {  // variants of S that occur in the sum
    std::vector<char> u(1u << __builtin_popcount(S), 0);
    for (int h = 0; h < H; ++h) u[pext8(hbits[h], S)] = 1;
    return u;
  };

  // producers, legs and readers
  std::vector<int> holder(P.n_slots, -1), reads(n_ops, 0), reader(n_ops, -1), ordinal(n_ops, -1);
  std::vector<int> src(4 * (size_t)n_ops, -1);
  std::vector<uint32_t> legs(n_ops, 0);
  int n_amp = 0;
  for (int i = 0; i < n_ops; ++i) {
    const Op& op = P.ops[i];
    const int n_in = op.type == OP_EXT ? 0 : op.n_in;
    for (int k = 0; k < n_in; ++k) {
      const int s = holder.at(op.in[k]);
      check(s >= 0, "slot read before it is written");
      src[4 * (size_t)i + k] = s;
      ++reads[s];
      reader[s] = i;
      legs[i] |= legs[s];
    }
    if (op.type == OP_EXT) legs[i] = 1u << op.leg;
    if (is_amp_op(op.type)) {
      check(legs[i] == all, "amplitude does not cover every leg");
      ordinal[i] = n_amp++;
    } else {
      holder.at(op.out) = i;
    }
  }
  for (int i = 0; i < n_ops; ++i)
    if (ordinal[i] >= 0) Q.flops += (double)H * op_flop_cost(P.ops[i]);
  check(n_amp < 0x10000 && weight.size() == (size_t)n_amp && row.size() == weight.size(),
        "diagram ordinals of 16 bits");

  // fused: read once, by a contraction, with n - 2 legs and at least two rounds
  std::vector<char> fused(n_ops, 0), stored(n_ops, 0);
  std::vector<int> fused_amp(n_ops, -1);  // of an amplitude: the current fused into it
  for (int i = 0; i < n_ops; ++i) {
    const Op& op = P.ops[i];
    if (is_amp_op(op.type)) continue;
    const bool current = op.type >= OP_JVV && op.type <= OP_JIO;
    if (current && __builtin_popcount(legs[i]) == n - 2 && reads[i] == 1 && P.ops[reader[i]].type == OP_ADOT &&
        src[4 * (size_t)reader[i]] == i && src[4 * (size_t)reader[i] + 1] != i) {
      fused[i] = 1;
      fused_amp[reader[i]] = i;
    } else if (reads[i] > 0) {
      stored[i] = 1;
    }
  }
  for (int i = 0; i < n_ops; ++i)
    for (int k = 0; k < 4; ++k) {
      const int s = src[4 * (size_t)i + k];
      check(s < 0 || stored[s] || (fused[s] && fused_amp[i] == s), "a fused current read elsewhere");
    }

  // area: resident values by level, then the block buffers
  int total = 0;
  for (int i = 0; i < n_ops; ++i)
    if (stored[i]) total += 1 << __builtin_popcount(legs[i]);
  const int block_legs = total > kResidentArea ? n - 3 : 99;
  std::vector<int> off(n_ops, -1), block(n_ops, -1);
  int top = 0, levels = 0;
  for (int lv = 1; lv < n; ++lv)
    for (int i = 0; i < n_ops; ++i) {
      if (!stored[i] || __builtin_popcount(legs[i]) != lv || lv == block_legs) continue;
      const int nv = 1 << lv, al = std::min(nv, 4);
      top = (top + al - 1) / al * al;
      off[i] = top;
      top += nv;
      levels = std::max(levels, lv);
    }
  check(block_legs == 99 || levels < block_legs, "a stored value above the block level");
  // blocks of leg sets: the larger sets first
  std::map<uint32_t, int> set_size;
  for (int i = 0; i < n_ops; ++i)
    if (stored[i] && __builtin_popcount(legs[i]) == block_legs) set_size[legs[i]] += 1 << block_legs;
  std::vector<std::pair<int, uint32_t>> order;
  for (auto& s : set_size) order.push_back({-s.second, s.first});
  std::sort(order.begin(), order.end());
  std::vector<int> fill;
  std::map<uint32_t, int> block_of;
  for (auto& o : order) {
    int b = -1;
    for (size_t k = 0; k < fill.size(); ++k)
      if (fill[k] - o.first <= kBlockArea) { b = (int)k; break; }
    if (b < 0) { b = (int)fill.size(); fill.push_back(0); }
    block_of[o.second] = b;
    fill[b] -= o.first;
  }
  const int n_blocks = (int)fill.size();
  int cap[2] = {0, 0};
  for (int b = 0; b < n_blocks; ++b) cap[b & 1] = std::max(cap[b & 1], fill[b]);
  top = (top + 3) / 4 * 4;
  const int buf[2] = {top, top + cap[0]};
  {
    std::vector<int> at(n_blocks, 0);
    for (int i = 0; i < n_ops; ++i) {
      if (!stored[i] || __builtin_popcount(legs[i]) != block_legs) continue;
      const int b = block_of[legs[i]];
      block[i] = b;
      off[i] = buf[b & 1] + at[b];
      at[b] += 1 << block_legs;
    }
  }
  Q.area = top + cap[0] + cap[1];
  check(Q.area <= max_area && Q.area <= 65535, "the area does not fit");

  // phases: levels 1 .. levels, block 0's values, then one per block (its
  // units and the next block's values); without blocks one consuming phase
  const int first_use = levels + (n_blocks > 0 ? 1 : 0);
  const int n_phases = first_use + std::max(1, n_blocks);
  std::vector<Costed> units;
  auto put = [&](const void* p, size_t bytes) {
    const size_t o = Q.rec.size();
    Q.rec.resize(o + bytes / 4);
    std::memcpy(Q.rec.data() + o, p, bytes);
  };
  auto here = [&] { return (uint32_t)(Q.rec.size() / 4); };
  auto phase_of_blocks = [&](std::initializer_list<int> values) {
    int ph = -1;
    for (int s : values) {
      if (s < 0 || block[s] < 0) continue;
      const int p = first_use + block[s];
      check(ph < 0 || ph == p, "a unit reads two blocks");
      ph = p;
    }
    return ph;
  };

  // PRODUCE
  {
    std::map<std::pair<int, int>, std::vector<PhItem>> items;  // (phase, op type)
    for (int i = 0; i < n_ops; ++i) {
      if (!stored[i]) continue;
      const Op& op = P.ops[i];
      const int ph = block[i] >= 0 ? (block[i] == 0 ? levels : first_use + block[i] - 1)
                                   : __builtin_popcount(legs[i]) - 1;
      const std::vector<char> u = used(legs[i]);
      const int n_in = op.type == OP_EXT ? 0 : op.n_in;
      for (int v = 0; v < (int)u.size(); ++v) {
        if (!u[v]) continue;
        const uint32_t lam = pdep8(v, legs[i]);
        Q.flops += op_flop_cost(op);
        PhItem it{};
        it.out = (uint16_t)(off[i] + v);
        for (int k = 0; k < n_in; ++k) {
          const int s = src[4 * (size_t)i + k];
          check(block[s] < 0, "a stored value reads a block value");
          it.in[k] = (uint16_t)(off[s] + pext8(lam, legs[s]));
        }
        switch (op.type) {
          case OP_EXT: it.x = (uint8_t)(op.leg | (lam >> op.leg & 1u) << 4); break;
          case OP_JVV: it.r[0] = (uint8_t)op.min[0]; it.r[1] = (uint8_t)op.min[1]; it.r[2] = (uint8_t)op.mout; break;
          case OP_JGGG: case OP_FVI: case OP_FVO: case OP_JIO: it.r[2] = (uint8_t)op.mout; break;
          case OP_PVVV: for (int k = 0; k < 3; ++k) it.r[k] = (uint8_t)op.min[k]; break;
          case OP_PGGGG: break;
          case OP_PIOV: it.x = (uint8_t)op.leg; break;
          default: check(false, "unknown op");
        }
        items[{ph, op.type}].push_back(it);
      }
    }
    for (auto& g : items)
      for (size_t b = 0; b < g.second.size(); b += 64) {
        const size_t k = std::min<size_t>(64, g.second.size() - b);
        Costed c{};
        c.u.type = PH_PRODUCE;
        c.u.op = (uint8_t)g.first.second;
        c.u.n = (uint16_t)k;
        c.u.rec = here();
        put(&g.second[b], k * sizeof(PhItem));
        c.cost = 40 + 140.0 * (double)((k + 31) / 32);
        c.phase = g.first.first;
        units.push_back(c);
      }
  }

  const int passes = (H + 31) / 32;
  std::vector<int> generic;
  // OUTER: contractions of stored free wavefunctions with stored partials
  {
    struct Key {
      uint32_t sf;
      int plain, ph;
      bool operator<(const Key& o) const { return std::tie(sf, plain, ph) < std::tie(o.sf, o.plain, o.ph); }
    };
    std::map<Key, std::map<int, std::map<int, int>>> groups;  // -> partial -> free -> amplitude op
    for (int i = 0; i < n_ops; ++i) {
      const Op& op = P.ops[i];
      if (!is_amp_op(op.type) || fused_amp[i] >= 0) continue;
      const int f = src[4 * (size_t)i], p = src[4 * (size_t)i + 1];
      if (op.type != OP_ADOT || (legs[f] & legs[p]) != 0) { generic.push_back(i); continue; }
      auto& slot = groups[{legs[f], (int)(op.leg & 1u), phase_of_blocks({f, p})}][p];
      if (slot.count(f)) generic.push_back(i);
      else slot[f] = i;
    }
    for (auto& g : groups) {
      // up to four partials with the same free wavefunctions share a unit
      std::map<std::vector<int>, std::vector<int>> same;
      for (auto& p : g.second) {
        std::vector<int> fs;
        for (auto& f : p.second) fs.push_back(f.first);
        same[fs].push_back(p.first);
      }
      for (auto& s : same)
        for (size_t p0 = 0; p0 < s.second.size(); p0 += kPhPartials) {
          const int np = (int)std::min<size_t>(kPhPartials, s.second.size() - p0);
          for (size_t f0 = 0; f0 < s.first.size(); f0 += kPhFree) {
            const int nf = (int)std::min<size_t>(kPhFree, s.first.size() - f0);
            Costed c{};
            c.u.type = PH_OUTER;
            c.u.op = (uint8_t)g.first.plain;
            c.u.n = (uint16_t)nf;
            c.u.rec = here();
            c.u.sf = (uint8_t)g.first.sf;
            c.u.sp = (uint8_t)(all & ~g.first.sf);
            c.u.np = (uint8_t)np;
            PhOuterHead hd{};
            for (int k = 0; k < 4; ++k) hd.p[k] = 32u * (uint32_t)off[s.second[p0 + std::min(k, np - 1)]];
            put(&hd, sizeof hd);
            for (int q = 0; q < nf; ++q) {
              const int f = s.first[f0 + q];
              PhOuterRec r{};
              r.f = 32u * (uint32_t)off[f];
              for (int k = 0; k < 4; ++k) r.d[k] = kPhNone;
              for (int k = 0; k < np; ++k) {
                const int a = g.second[s.second[p0 + k]][f];
                r.d[k] = (uint32_t)row[ordinal[a]];
                r.w[k] = weight[ordinal[a]];
              }
              put(&r, sizeof r);
            }
            c.cost = 60 + nf * (10 + 30.0 * np);
            c.phase = g.first.ph;
            for (int j = 0; j < passes; ++j) {
              c.u.pass = (uint8_t)j;
              units.push_back(c);
            }
          }
        }
    }
  }
  // FUSED
  {
    std::map<uint32_t, int> set_index;
    std::map<std::tuple<int, uint32_t, int>, std::vector<int>> groups;  // (phase, legs, op type) -> amplitude ops
    for (int i = 0; i < n_ops; ++i) {
      if (fused_amp[i] < 0) continue;
      const int t = fused_amp[i], p = src[4 * (size_t)i + 1];
      check((legs[t] & legs[p]) == 0, "fused current and partial share legs");
      check((P.ops[i].leg & 1u) == ((P.ops[t].type == OP_FVI || P.ops[t].type == OP_FVO) ? 1u : 0u), "contraction of a fused current");
      int ph = block[p] >= 0 ? first_use + block[p] : -1;
      const int n_in = P.ops[t].n_in;
      for (int k = 0; k < n_in; ++k) {
        const int q = phase_of_blocks({src[4 * (size_t)t + k]});
        check(q < 0 || ph < 0 || q == ph, "a unit reads two blocks");
        if (q >= 0) ph = q;
      }
      groups[{ph, legs[t], (int)P.ops[t].type}].push_back(i);
    }
    for (auto& g : groups) {
      // currents with the same partial follow each other
      std::stable_sort(g.second.begin(), g.second.end(),
                       [&](int x, int y) { return src[4 * (size_t)x + 1] < src[4 * (size_t)y + 1]; });
      const uint32_t S = std::get<1>(g.first), SP = all & ~S;
      const std::vector<char> u = used(S);
      std::vector<int> vs;
      for (int v = 0; v < (int)u.size(); ++v)
        if (u[v]) vs.push_back(v);
      check(!vs.empty() && vs.size() <= 32, "variants of a fused current");
      for (int i : g.second) Q.flops += (double)vs.size() * op_flop_cost(P.ops[fused_amp[i]]);
      int lg = 0;
      while ((1 << lg) < (int)vs.size()) ++lg;
      if (!set_index.count(S)) {
        PhSet T;
        std::memset(&T, 0, sizeof T);
        for (auto& r : T.uh)
          for (uint16_t& x : r) x = kPhNoPair;
        std::vector<int> legs_of;
        for (int l = 0; l < n; ++l)
          if (S >> l & 1u) legs_of.push_back(l);
        for (int lane = 0; lane < 32; ++lane) {
          const int i = lane & ((1 << lg) - 1);
          const bool on = i < (int)vs.size();
          const int v = on ? vs[i] : vs[0];
          T.v[lane] = (uint8_t)v;
          for (uint32_t m = 0; m < 32; ++m) T.sub[m][lane] = (uint16_t)(32u * pext8((uint32_t)v, m));
          int r = 0;
          for (int h = 0; h < H && on; ++h)
            if ((int)pext8(hbits[h], S) == v) {
              check(r < kPhRounds, "rounds of a fused current");
              T.uh[r++][lane] = (uint16_t)(pext8(hbits[h], SP) | (uint32_t)h << 8);
            }
        }
        set_index[S] = (int)Q.sets.size();
        Q.sets.push_back(T);
      }
      int rounds = 0;
      for (int lane = 0; lane < 32; ++lane)
        while (rounds < kPhRounds && Q.sets[set_index[S]].uh[rounds][lane] != kPhNoPair) ++rounds;
      const int per_pass = 32 >> lg;
      const size_t most = (size_t)std::max(8, 4 * per_pass);
      for (size_t b = 0; b < g.second.size(); b += most) {
        const size_t k = std::min(most, g.second.size() - b);
        Costed c{};
        c.u.type = PH_FUSED;
        c.u.op = (uint8_t)std::get<2>(g.first);
        c.u.n = (uint16_t)k;
        c.u.rec = here();
        c.u.set = (uint16_t)set_index[S];
        c.u.lanes = (uint8_t)lg;
        c.u.rounds = (uint8_t)rounds;
        for (size_t q = 0; q < k; ++q) {
          const int a = g.second[b + q], t = fused_amp[a];
          const Op& op = P.ops[t];
          PhFusedRec r{};
          for (int j = 0; j < op.n_in; ++j) {
            const int s = src[4 * (size_t)t + j];
            r.in[j] = 32u * (uint32_t)off[s];
            r.m[j] = 64u * pext8(legs[s], S);
          }
          if (op.type == OP_JVV) { r.r[0] = 32u * op.min[0]; r.r[1] = 32u * op.min[1]; }
          r.r[2] = 32u * op.mout;
          r.p = 32u * (uint32_t)off[src[4 * (size_t)a + 1]];
          r.d = (uint32_t)row[ordinal[a]];
          r.w = weight[ordinal[a]];
          put(&r, sizeof r);
        }
        c.cost = 150 + (120.0 + 40.0 * rounds) * (double)((k + per_pass - 1) / per_pass);
        c.phase = std::get<0>(g.first);
        units.push_back(c);
      }
    }
  }
  // GENERIC
  {
    std::map<int, std::vector<int>> groups;
    for (int i : generic) {
      int ph = -1;
      for (int k = 0; k < P.ops[i].n_in; ++k) {
        const int q = phase_of_blocks({src[4 * (size_t)i + k]});
        check(q < 0 || ph < 0 || q == ph, "a unit reads two blocks");
        if (q >= 0) ph = q;
      }
      groups[ph].push_back(i);
    }
    for (auto& g : groups)
      for (size_t b = 0; b < g.second.size(); b += 12) {
        const size_t k = std::min<size_t>(12, g.second.size() - b);
        Costed c{};
        c.u.type = PH_GENERIC;
        c.u.n = (uint16_t)k;
        c.u.rec = here();
        for (size_t q = 0; q < k; ++q) {
          const Op& op = P.ops[g.second[b + q]];
          PhGenericRec r{};
          r.type = op.type;
          r.flags = (uint8_t)op.leg;
          r.d = (uint16_t)row[ordinal[g.second[b + q]]];
          for (int j = 0; j < op.n_in; ++j) {
            const int s = src[4 * (size_t)g.second[b + q] + j];
            r.in[j] = (uint16_t)off[s];
            r.m[j] = (uint8_t)legs[s];
          }
          for (int j = 0; j < 3; ++j) r.r[j] = (uint8_t)op.min[j];
          r.w = weight[ordinal[g.second[b + q]]];
          put(&r, sizeof r);
        }
        c.cost = 60 + 150.0 * (double)k;
        c.phase = g.first;
        for (int j = 0; j < passes; ++j) {
          c.u.pass = (uint8_t)j;
          units.push_back(c);
        }
      }
  }

  // units that read no block fill the lighter consuming phases
  std::vector<double> load(n_phases, 0);
  for (auto& c : units) {
    Q.cost += c.cost;
    if (c.phase >= 0) load[c.phase] += c.cost;
  }
  for (auto& c : units)
    if (c.phase < 0) {
      int best = first_use;
      for (int p = first_use; p < n_phases; ++p)
        if (load[p] < load[best]) best = p;
      c.phase = best;
      load[best] += c.cost;
    }
  // each phase's units onto kPhWarps lists, the costly ones first, each to the
  // list with the least work; the warps of a CTA take lists w, w + W, ...
  std::stable_sort(units.begin(), units.end(), [](const Costed& a, const Costed& b) {
    return a.phase != b.phase ? a.phase < b.phase : a.cost > b.cost;
  });
  Q.phases = n_phases;
  for (int p = 0, i = 0; p < n_phases; ++p) {
    std::vector<std::vector<PhUnit>> list(kPhWarps);
    std::vector<double> work(kPhWarps, 0.0);
    for (; i < (int)units.size() && units[i].phase == p; ++i) {
      const int l = (int)(std::min_element(work.begin(), work.end()) - work.begin());
      list[l].push_back(units[i].u);
      work[l] += units[i].cost;
    }
    for (auto& l : list) {
      Q.units.insert(Q.units.end(), l.begin(), l.end());
      Q.list_end.push_back((int)Q.units.size());
    }
  }
  return Q;
}

}  // namespace mea
