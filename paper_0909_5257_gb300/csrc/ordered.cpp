// Ordered-recursion layout of a process (see ordered.h).
#include "ordered.h"

#include <algorithm>
#include <cstring>
#include <map>
#include <stdexcept>
#include <string>
#include <tuple>

namespace mea {
namespace {

typedef std::vector<int> Word;  // letters

void check(bool ok, const char* why) {
  if (!ok) throw LayoutError(std::string("ordered recursion: ") + why);
}

struct Val {
  int off = 0;    // 16-byte units
  int nb = 0;     // helicity bits
  int level = 0;  // stage level it is made in
  uint32_t legs = 0;
};

struct Item {
  OrdStage st;
  int level;
  std::vector<uint64_t> rec;
};

struct Build {
  const Program& P;
  OrdProgram& Q;
  std::vector<uint32_t> letter_legs;
  std::vector<int> letter_bits;
  std::vector<Val> letter_val;
  std::map<Word, Val> gluon;
  std::map<std::tuple<int, int, Word>, Val> quark;  // (barred, leg, word)
  std::map<std::pair<int, int>, Val> ext_q;         // (barred, leg)
  std::vector<Item> items;

  explicit Build(const Program& p, OrdProgram& q) : P(p), Q(q) {}

  int row(uint32_t legs) {
    for (size_t r = 0; r < P.masks.size(); ++r)
      if (P.masks[r] == legs) {
        check(r < 256, "event-table row");
        return (int)r;
      }
    check(false, "a momentum outside the event table");
    return 0;
  }
  int alloc(int variants, int doubles) {
    const int o = Q.area / 2;
    check(o < 65536, "area offset");
    Q.area += variants * doubles;
    return o;
  }
  static uint64_t pack(int off, int row, int sh, int nb, int flags, int pad = 0) {
    check(off < 65536 && row < 256 && sh < 256 && nb < 256, "field");
    return (uint64_t)off | (uint64_t)row << 16 | (uint64_t)sh << 24 | (uint64_t)nb << 32 | (uint64_t)flags << 40 | (uint64_t)pad << 48;
  }
  void emit(int type, int k, int nb, bool full, int level, std::vector<uint64_t> rec) {
    Item it;
    std::memset(&it.st, 0, sizeof it.st);
    it.st.type = (uint8_t)type;
    it.st.k = (uint8_t)k;
    it.st.nb = (uint8_t)nb;
    it.st.full = full ? 1 : 0;
    it.level = level;
    it.rec = std::move(rec);
    items.push_back(std::move(it));
  }

  int bits(const Word& w, size_t i, size_t j) const {
    int b = 0;
    for (size_t k = i; k < j; ++k) b += letter_bits[w[k]];
    return b;
  }
  uint32_t legs_of(const Word& w) const {
    uint32_t m = 0;
    for (int x : w) m |= letter_legs[x];
    return m;
  }
  bool conserved(const Word& w) const {  // gluon legs only
    for (int x : w)
      if (letter_legs[x] & (letter_legs[x] - 1)) return false;
    return true;
  }
  // stored form of a word: reversed words of one-bit letters are equal up to the sign (-1)^(k-1)
  Word canonical(const Word& w, bool& rev) const {
    rev = false;
    if (!conserved(w)) return w;
    for (int x : w)
      if (letter_bits[x] != 1) return w;
    Word r(w.rbegin(), w.rend());
    if (r < w) { rev = true; return r; }
    return w;
  }

  int add_gluon_letter(int leg, int nbits, int fixed) {
    Val v;
    v.nb = nbits;
    v.legs = 1u << leg;
    v.off = alloc(1 << nbits, 8);
    emit(ORD_EXT_G, 1, nbits, false, 0, {pack(v.off, leg, 0, nbits, fixed)});
    letter_legs.push_back(v.legs);
    letter_bits.push_back(nbits);
    letter_val.push_back(v);
    return (int)letter_val.size() - 1;
  }
  Val external_quark(int barred, int leg, bool both) {
    auto key = std::make_pair(barred, leg);
    auto it = ext_q.find(key);
    if (it != ext_q.end()) {
      check(it->second.nb == (both ? 1 : 0), "a quark leg on both lines' forms");
      return it->second;
    }
    Val v;
    v.nb = both ? 1 : 0;
    v.legs = 1u << (leg % 100);
    v.off = alloc(1 << v.nb, 4);
    emit(ORD_EXT_Q, 0, v.nb, false, 0, {pack(v.off, leg % 100, 0, 0, (barred ? 1 : 0) | (both ? 2 : 0))});
    return ext_q[key] = v;
  }

  // reference to letters i .. j - 1 of w; `low`: bits behind the word's last letter in the pattern
  OrdRef none{};
  uint64_t sub(const Word& w, size_t i, size_t j, int low, int& level) {
    const Word s(w.begin() + i, w.begin() + j);
    bool rev = false;
    const Val v = get(canonical(s, rev));
    level = std::max(level, v.level);
    const bool neg = rev && s.size() % 2 == 0;
    return pack(v.off, row(v.legs), bits(w, j, w.size()) + low, v.nb, (rev ? 1 : 0) | (neg ? 2 : 0));
  }
  std::vector<uint64_t> subs(const Word& w, int& level, size_t longest) {
    std::vector<uint64_t> r;
    for (size_t i = 0; i < w.size(); ++i)
      for (size_t j = i + 1; j <= w.size(); ++j) r.push_back(j - i <= longest && j - i < w.size() ? sub(w, i, j, 0, level) : 0);
    return r;
  }
  Val get(const Word& w) {
    if (w.size() == 1) return letter_val[w[0]];
    auto it = gluon.find(w);
    if (it != gluon.end()) return it->second;
    int level = 0;
    std::vector<uint64_t> s = subs(w, level, w.size());
    Val v;
    v.nb = bits(w, 0, w.size());
    v.legs = legs_of(w);
    v.level = level + 1;
    v.off = alloc(1 << v.nb, 8);
    s.insert(s.begin(), pack(v.off, row(v.legs), 0, 0, 0));
    emit(ORD_G, (int)w.size(), v.nb, !conserved(w), v.level, s);
    return gluon[w] = v;
  }
  // quark word of a line; both: the line's chirality is the pattern's top bit
  // (leg + 100: a leg's right-handed form beside its form of both chiralities)
  Val get_quark(int barred, int leg, const Word& w, bool both) {
    if (w.empty()) return external_quark(barred, leg, both);
    auto key = std::make_tuple(barred, leg, w);
    auto it = quark.find(key);
    if (it != quark.end()) return it->second;
    int level = 0;
    std::vector<uint64_t> r{0};
    const size_t k = w.size();
    for (size_t i = 1; i <= k; ++i) {  // gluon piece of i letters next to the vertex
      if (!barred) {
        r.push_back(sub(w, 0, i, 0, level));
        const Val s = get_quark(0, leg, Word(w.begin() + i, w.end()), both);
        level = std::max(level, s.level);
        r.push_back(pack(s.off, 0, 0, s.nb, 0));
      } else {
        r.push_back(sub(w, k - i, k, 0, level));
        const Val s = get_quark(1, leg, Word(w.begin(), w.end() - i), both);
        level = std::max(level, s.level);
        r.push_back(pack(s.off, 0, bits(w, k - i, k), s.nb, 0));
      }
    }
    Val v;
    v.nb = bits(w, 0, k) + (both ? 1 : 0);
    v.legs = legs_of(w) | 1u << (leg % 100);
    v.level = level + 1;
    v.off = alloc(1 << v.nb, 4);
    r[0] = pack(v.off, row(v.legs), 0, 0, both ? 4 : 0);
    emit(barred ? ORD_BAR : ORD_PSI, (int)k, v.nb, false, v.level, r);
    return quark[key] = v;
  }
  uint64_t close(int f, int z, int xnb, bool left, bool rev, bool neg) {
    check(f < 65536 && z < 65536, "closing");
    return (uint64_t)f | (uint64_t)z << 16 | (uint64_t)xnb << 32 | (uint64_t)(left ? 1 : 0) << 40 | (uint64_t)(rev ? 1 : 0) << 48 |
           (uint64_t)(neg ? 1 : 0) << 56;
  }
};

constexpr int kLevelAmp = 1000;  // amplitudes, then what is added to them

uint32_t word_pattern(const Build& B, const Word& w, const std::vector<uint32_t>& letter_pattern) {
  uint32_t v = 0;
  for (int x : w) v = v << B.letter_bits[x] | letter_pattern[x];
  return v;
}

}  // namespace

OrdProgram build_ordered(const Program& P, const ColourBase* known) {
  OrdProgram Q;
  Build B(P, Q);
  const int n = P.n_ext;
  std::vector<int> gl, psi, bar;
  for (int l = 0; l < n; ++l) (P.leg_type[l] == 0 ? gl : P.leg_type[l] == 1 ? psi : bar).push_back(l);
  const int ng = (int)gl.size();
  Q.norm = 2.0 / (double)P.cf_den;
  std::vector<std::vector<uint16_t>> fidx;  // [a][h]

  if (P.family == FAM_GLUON) {
    check(P.root == n - 1, "root leg");
    const ColourBase base = known ? *known : find_colour_base(P);
    const int n_base = base.mb;
    const std::vector<uint16_t>&kk_index = base.index, &kk_term = base.term;
    const int k = n - 2;  // letters of a fused word
    for (int l = 0; l < n - 1; ++l) B.add_gluon_letter(l, l == 0 ? 0 : 1, 0);
    const int root = B.add_gluon_letter(n - 1, 1, 0);
    const Val eps = B.letter_val[root];
    // [J(x), eps] of every letter for both root polarisations
    std::vector<Val> z(n - 1);
    for (int x = 0; x < n - 1; ++x) {
      const Val& v = B.letter_val[x];
      z[x].nb = v.nb + 1;
      z[x].off = B.alloc(1 << z[x].nb, 8);
      B.emit(ORD_Z, 0, z[x].nb, false, 1,
             {Build::pack(z[x].off, 0, 0, 0, 0), Build::pack(v.off, B.row(v.legs), 0, 0, 0), Build::pack(eps.off, B.row(eps.legs), 0, 0, 0)});
    }
    Word rest;
    for (int l = 1; l < n - 1; ++l) rest.push_back(l);
    std::vector<Word> words;
    do {
      Word w{0};
      w.insert(w.end(), rest.begin(), rest.end());
      words.push_back(w);
    } while (std::next_permutation(rest.begin(), rest.end()));
    check((int)words.size() == n_base, "base of the ordered traces");
    Q.n_colour = (int)words.size();
    const int per = 1 << (n - 1);
    std::map<Word, std::vector<uint64_t>> closings;  // fused word -> closings
    for (size_t a = 0; a < words.size(); ++a) {
      const Word& w = words[a];
      int level = 0;
      std::vector<uint64_t> r = B.subs(w, level, (size_t)k - 1);
      r.insert(r.begin(), Build::pack(eps.off, 0, 0, 0, 0));
      r.insert(r.begin(), Build::pack((int)a * per, 0, 0, 0, 0));
      B.emit(ORD_GA, n - 1, n - 2, false, kLevelAmp, r);
      for (int left = 0; left < 2; ++left) {  // letter left or right of the fused word
        const Word s(w.begin() + left, w.end() - (1 - left));
        const int x = left ? w.front() : w.back();
        bool rev = false;
        const Word c = B.canonical(s, rev);
        // eps.[u, v] = u.[v, eps] = -v.[u, eps]
        const bool neg = (left != 0) != (rev && s.size() % 2 == 0);
        closings[c].push_back(B.close((int)a * per, z[x].off, B.letter_bits[x], left != 0, rev, neg));
      }
    }
    for (auto& c : closings) {
      int level = 0;
      std::vector<uint64_t> r = B.subs(c.first, level, c.first.size());
      r.insert(r.begin(), Build::pack(0, B.row(B.legs_of(c.first)), (int)c.second.size(), 0, 1));
      r.insert(r.end(), c.second.begin(), c.second.end());
      B.emit(ORD_GF, k, B.bits(c.first, 0, c.first.size()), false, kLevelAmp + 1 + (c.first[0] == 0 ? 0 : 1), r);
    }
    Q.n_f = Q.n_colour * per;
    Q.norm *= 4.0;  // coefficient 2 of the ordered trace Tr(T^r T^w)
    fidx.resize(Q.n_colour);
    for (int h = 0; h < P.n_hel; ++h) {
      const int8_t* lam = &P.hel[(size_t)h * n];
      if (lam[0] > 0) continue;
      std::vector<uint32_t> lp(n);
      for (int l = 0; l < n; ++l) lp[l] = l == 0 ? 0 : lam[l] > 0;
      for (size_t a = 0; a < words.size(); ++a)
        fidx[a].push_back((uint16_t)(a * per + 2 * word_pattern(B, words[a], lp) + lp[n - 1]));
      Q.range.push_back(0);
      Q.range.push_back(Q.n_colour);
    }
    // colour matrix of the base: R^T K R, R the signed sums of the other orderings
    const int m = P.n_jamp;
    check(n_base == m || (int)kk_index.size() == 3 * (m - n_base), "sums of the base");
    std::vector<std::vector<std::pair<int, double>>> R(m);
    for (int a = 0; a < m; ++a) {
      if (a < n_base) { R[a].push_back({a, 1.0}); continue; }
      const uint16_t* ix = &kk_index[3 * (a - n_base)];
      for (int b = ix[0]; b < ix[2]; ++b) R[a].push_back({kk_term[b], b < ix[1] ? 1.0 : -1.0});
    }
    Q.kmat.assign((size_t)n_base * n_base, 0.0);
    for (int a = 0; a < m; ++a)
      for (int b = 0; b < m; ++b) {
        const double kv = (double)P.cf_jamp[(size_t)a * m + b];
        if (kv == 0.0) continue;
        for (auto& x : R[a])
          for (auto& y : R[b]) Q.kmat[(size_t)x.first * n_base + y.first] += x.second * y.second * kv;
      }
  } else if (P.family == FAM_ONE_LINE) {
    const int y = psi[0], root = P.root;
    std::map<int, int> letter;
    for (int l : gl) letter[l] = B.add_gluon_letter(l, 1, 0);
    const Val rowv = B.external_quark(1, root, false), colv = B.external_quark(0, y, false);
    Val z;
    z.off = B.alloc(1, 8);
    B.emit(ORD_Z, 0, 0, false, 1, {Build::pack(z.off, 0, 0, 0, 1), Build::pack(rowv.off, 0, 0, 0, 0), Build::pack(colv.off, 0, 0, 0, 0)});
    Q.n_colour = P.n_jamp;
    const int per = 1 << ng;
    std::vector<Word> words;
    for (const auto& c : P.basis) {
      Word w;
      for (int l : c[0].first) w.push_back(letter.at(l));
      words.push_back(w);
    }
    std::map<Word, std::vector<uint64_t>> g_close, q_close;
    for (size_t a = 0; a < words.size(); ++a) {
      const Word& w = words[a];
      int level = 0;
      std::vector<uint64_t> r{0, Build::pack(rowv.off, 0, 0, 0, 0)};
      int splits = 0;
      for (size_t i = 2; i < w.size(); ++i, ++splits) {
        r.push_back(B.sub(w, 0, i, 0, level));
        const Val s = B.get_quark(0, y, Word(w.begin() + i, w.end()), false);
        r.push_back(Build::pack(s.off, 0, 0, s.nb, 0));
      }
      r[0] = Build::pack((int)a * per, 0, splits, 0, 0);
      while (r.size() < 2 + 2 * (size_t)std::max(0, ng - 2)) r.push_back(0);
      B.emit(ORD_PA, ng, ng, false, kLevelAmp, r);
      bool rev = false;
      const Word c = B.canonical(w, rev);
      g_close[c].push_back(B.close((int)a * per, z.off, 0, false, rev, rev && ng % 2 == 0));
      q_close[Word(w.begin() + 1, w.end())].push_back(
          B.close((int)a * per, B.letter_val[w[0]].off, B.letter_bits[w[0]], true, false, false));
    }
    for (auto& c : g_close) {
      int level = 0;
      std::vector<uint64_t> r = B.subs(c.first, level, c.first.size());
      r.insert(r.begin(), Build::pack(0, B.row(B.legs_of(c.first)), (int)c.second.size(), 0, 0));
      r.insert(r.end(), c.second.begin(), c.second.end());
      B.emit(ORD_GF, ng, ng, false, kLevelAmp + 1, r);
    }
    for (auto& c : q_close) {
      int level = 0;
      std::vector<uint64_t> r{Build::pack(0, B.row(B.legs_of(c.first) | 1u << y), (int)c.second.size(), 0, 0),
                              Build::pack(rowv.off, 0, 0, 0, 0)};
      const Word& w = c.first;
      for (size_t i = 1; i <= w.size(); ++i) {
        r.push_back(B.sub(w, 0, i, 0, level));
        const Val s = B.get_quark(0, y, Word(w.begin() + i, w.end()), false);
        r.push_back(Build::pack(s.off, 0, 0, s.nb, 0));
      }
      r.insert(r.end(), c.second.begin(), c.second.end());
      B.emit(ORD_PF, ng - 1, ng - 1, false, kLevelAmp + 2, r);
    }
    Q.n_f = Q.n_colour * per;
    fidx.resize(Q.n_colour);
    // the right-handed quark line: u (incoming quark) of helicity +1, v (outgoing antiquark) of -1
    const int want = P.incoming[y] ? 1 : -1;
    for (int h = 0; h < P.n_hel; ++h) {
      const int8_t* lam = &P.hel[(size_t)h * n];
      if (lam[y] != want) continue;
      std::vector<uint32_t> lp(ng);
      for (int l : gl) lp[letter[l]] = lam[l] > 0;
      for (size_t a = 0; a < words.size(); ++a) fidx[a].push_back((uint16_t)(a * per + word_pattern(B, words[a], lp)));
      Q.range.push_back(0);
      Q.range.push_back(Q.n_colour);
    }
  } else {
    const int root = P.root;
    std::map<int, int> letter;
    for (int l : gl) letter[l] = B.add_gluon_letter(l, 1, 0);
    Q.n_colour = P.n_jamp;
    const int per = 1 << (ng + 1);
    std::map<std::tuple<int, int, Word, Word>, int> composite;  // (y2, z2, t, u) -> letter
    std::vector<Word> words;
    std::vector<int> second(Q.n_colour);  // letter of the second line's current
    std::vector<int> pairing(Q.n_colour);
    for (size_t a = 0; a < P.basis.size(); ++a) {
      const auto& c = P.basis[a];
      const int y = c[0].second[1], z2 = c[1].second[0], y2 = c[1].second[1];
      Word t, u;
      bool after = false;
      for (int l : c[1].first) {
        if (l == 100) after = true;
        else (after ? u : t).push_back(letter.at(l));
      }
      auto key = std::make_tuple(y2, z2, t, u);
      auto it = composite.find(key);
      if (it == composite.end()) {
        const Val r = B.get_quark(1, z2, t, true), s = B.get_quark(0, y2, u, true);
        Val v;
        v.nb = 1 + B.bits(t, 0, t.size()) + B.bits(u, 0, u.size());
        v.legs = r.legs | s.legs;
        v.level = std::max(r.level, s.level) + 1;
        v.off = B.alloc(1 << v.nb, 8);
        B.emit(ORD_X, 0, v.nb, false, v.level,
               {Build::pack(v.off, B.row(v.legs), 0, 0, 4), Build::pack(r.off, 0, s.nb - 1, r.nb, 0), Build::pack(s.off, 0, 0, s.nb, 0)});
        B.letter_legs.push_back(v.legs);
        B.letter_bits.push_back(v.nb);
        B.letter_val.push_back(v);
        it = composite.emplace(key, (int)B.letter_val.size() - 1).first;
      }
      Word w;
      for (int l : c[0].first) w.push_back(l == 100 ? it->second : letter.at(l));
      words.push_back(w);
      second[a] = it->second;
      pairing[a] = y == psi[0] ? 0 : 1;
    }
    const int k_max = ng + 1;
    for (size_t a = 0; a < words.size(); ++a) {
      const Word& w = words[a];
      const int y = P.basis[a][0].second[1];
      const Val rowv = B.external_quark(1, root, false);
      int level = 0;
      std::vector<uint64_t> r{Build::pack((int)a * per, 0, (int)w.size(), 0, 0), Build::pack(rowv.off, 0, 0, 0, 0)};
      for (size_t i = 1; i <= w.size(); ++i) {
        r.push_back(B.sub(w, 0, i, 0, level));
        // the first line's quark; the second line's form of the same leg has both chiralities
        const Val s = B.get_quark(0, y + 100, Word(w.begin() + i, w.end()), false);
        r.push_back(Build::pack(s.off, 0, 0, s.nb, 0));
      }
      while (r.size() < 2 + 2 * (size_t)k_max) r.push_back(0);
      B.emit(ORD_PA, 0, ng + 1, false, kLevelAmp, r);
    }
    Q.n_f = Q.n_colour * per;
    fidx.resize(Q.n_colour);
    int begin[3] = {0, 0, Q.n_colour};
    for (int a = 0; a < Q.n_colour; ++a)
      if (pairing[a] == 0) begin[1] = a + 1;
    for (int a = 0; a < Q.n_colour; ++a) check((a >= begin[1]) == (pairing[a] == 1), "order of the pairings");
    const bool two = begin[1] > 0 && begin[1] < Q.n_colour;
    // second line right-handed: both pairings; left-handed: one of them
    for (int cfg = 0; cfg < (two ? 3 : 2); ++cfg)
      for (uint32_t g = 0; g < (1u << ng); ++g) {
        std::vector<uint32_t> lp(B.letter_val.size(), 0);
        for (int i = 0; i < ng; ++i) lp[letter[gl[i]]] = g >> i & 1u;
        for (auto& c : composite) {
          uint32_t v = cfg > 0 ? 1u : 0u;
          for (int x : std::get<2>(c.first)) v = v << 1 | lp[x];
          for (int x : std::get<3>(c.first)) v = v << 1 | lp[x];
          lp[c.second] = v;
        }
        for (int a = 0; a < Q.n_colour; ++a) fidx[a].push_back((uint16_t)(a * per + word_pattern(B, words[a], lp)));
        Q.range.push_back(cfg < 2 || !two ? 0 : begin[1]);
        Q.range.push_back(cfg == 1 && two ? begin[1] : Q.n_colour);
      }
    // the exchanged pairing enters with the Fermi sign
    Q.kmat.resize((size_t)Q.n_colour * Q.n_colour);
    for (int a = 0; a < Q.n_colour; ++a)
      for (int b = 0; b < Q.n_colour; ++b)
        Q.kmat[(size_t)a * Q.n_colour + b] = (pairing[a] == pairing[b] ? 1.0 : -1.0) * (double)P.cf_jamp[(size_t)a * P.n_jamp + b];
  }
  Q.H = (int)Q.range.size() / 2;
  check(2 * Q.H == P.n_hel, "half of the helicity combinations");
  check(Q.n_f <= 65536, "amplitudes");
  if (Q.kmat.empty()) {
    check(P.n_jamp == Q.n_colour, "colour basis");
    for (int64_t v : P.cf_jamp) Q.kmat.push_back((double)v);
  }
  for (auto& f : fidx) Q.fidx.insert(Q.fidx.end(), f.begin(), f.end());

  // stages: items of one level and form
  std::stable_sort(B.items.begin(), B.items.end(), [](const Item& a, const Item& b) {
    return std::make_tuple(a.level, a.st.type, a.st.k, a.st.nb, a.st.full, a.rec.size()) <
           std::make_tuple(b.level, b.st.type, b.st.k, b.st.nb, b.st.full, b.rec.size());
  });
  auto same = [](const Item& a, const Item& b) {
    return a.level == b.level && a.st.type == b.st.type && a.st.k == b.st.k && a.st.nb == b.st.nb && a.st.full == b.st.full &&
           a.rec.size() == b.rec.size();
  };
  for (size_t i = 0; i < B.items.size();) {
    size_t j = i;
    while (j < B.items.size() && same(B.items[i], B.items[j])) ++j;
    OrdStage st = B.items[i].st;
    st.words = (uint16_t)(j - i);
    st.stride = (uint16_t)B.items[i].rec.size();
    st.rec = (uint32_t)Q.rec.size();
    for (size_t q = i; q < j; ++q) Q.rec.insert(Q.rec.end(), B.items[q].rec.begin(), B.items[q].rec.end());
    Q.level.push_back(B.items[i].level);
    Q.stages.push_back(st);
    i = j;
  }
  return Q;
}

}  // namespace mea
