// Base of a process's colour amplitudes (see colour_base.h).
#include "colour_base.h"

#include <algorithm>

namespace mea {

// Base of the rows of C (m x kd small integers): the first rows that no
// earlier ones generate, and the others as sums of them, by elimination
// modulo a prime on random combinations of the columns (checked exactly below).  Returns false unless the base is rows 0 .. mb - 1
// and every coefficient is 0, 1 or -1.
static bool find_base(const std::vector<int>& C, int m, int kd, int& mb, std::vector<std::vector<int>>& coef) {
  typedef unsigned long long u64;
  const u64 P = 2147483647ull;
  auto inv = [&](u64 a) {
    u64 r = 1, e = P - 2;
    for (; e; e >>= 1, a = a * a % P)
      if (e & 1) r = r * a % P;
    return r;
  };
  const int cols = m + 8;
  u64 seed = 0x9E3779B97F4A7C15ull;
  std::vector<u64> X((size_t)m * cols, 0), rnd(cols);
  for (int d = 0; d < kd; ++d) {
    for (u64& x : rnd) {  // a linear congruential sequence
      seed = seed * 6364136223846793005ull + 1442695040888963407ull;
      x = (seed >> 33) % P;
    }
    for (int a = 0; a < m; ++a) {
      const int c = C[(size_t)a * kd + d];
      if (!c) continue;
      const u64 cc = (u64)((c + (long long)P) % (long long)P);
      for (int j = 0; j < cols; ++j) X[(size_t)a * cols + j] = (X[(size_t)a * cols + j] + cc * rnd[j]) % P;
    }
  }
  std::vector<std::vector<u64>> B, T;  // reduced rows and what they are of the base rows
  std::vector<int> piv;
  mb = 0;
  coef.clear();
  for (int a = 0; a < m; ++a) {
    std::vector<u64> r(X.begin() + (size_t)a * cols, X.begin() + (size_t)(a + 1) * cols), c(m, 0);
    for (size_t b = 0; b < B.size(); ++b) {
      const u64 f = r[piv[b]];
      if (!f) continue;
      for (int j = 0; j < cols; ++j) r[j] = (r[j] + (P - f) * B[b][j]) % P;
      for (int j = 0; j < mb; ++j) c[j] = (c[j] + f * T[b][j]) % P;
    }
    int q = -1;
    for (int j = 0; j < cols && q < 0; ++j)
      if (r[j]) q = j;
    if (q >= 0) {
      if (a != mb) return false;  // the base is not a prefix
      const u64 iv = inv(r[q]);
      for (u64& x : r) x = x * iv % P;
      std::vector<u64> tb(m, 0);
      for (int j = 0; j < mb; ++j) tb[j] = (P - c[j]) % P * iv % P;
      tb[mb] = iv;
      B.push_back(r);
      T.push_back(tb);
      piv.push_back(q);
      ++mb;
    } else {
      std::vector<int> k(m, 0);
      for (int j = 0; j < mb; ++j) {
        if (c[j] == 1) k[j] = 1;
        else if (c[j] == P - 1) k[j] = -1;
        else if (c[j] != 0) return false;
      }
      coef.push_back(k);
    }
  }
  return true;
}

ColourBase find_colour_base(const Program& p) {
  ColourBase B;
  const int m = p.n_jamp;
  B.mb = m;
  int kd = 0;
  for (const Op& op : p.ops) kd += is_amp_op(op.type) ? 1 : 0;
  std::vector<int> C((size_t)m * kd, 0);
  int d = 0;
  for (const Op& op : p.ops) {
    if (!is_amp_op(op.type)) continue;
    for (uint32_t k = 0; k < op.col_count; ++k) {
      const ColEntry& c = p.col[op.col_begin + k];
      if (c.im != 0) return B;
      C[(size_t)c.alpha * kd + d] += c.re;
    }
    ++d;
  }
  int mb = 0;
  std::vector<std::vector<int>> coef;
  if (!find_base(C, m, kd, mb, coef) || mb >= m) return B;
  std::vector<uint16_t> index, term;
  for (int a = mb; a < m; ++a) {
    const std::vector<int>& k = coef[a - mb];
    std::vector<int> row(kd, 0);
    index.push_back((uint16_t)term.size());
    for (int sg : {1, -1}) {
      for (int b = 0; b < mb; ++b)
        if (k[b] == sg) {
          term.push_back((uint16_t)b);
          for (int x = 0; x < kd; ++x) row[x] += sg * C[(size_t)b * kd + x];
        }
      index.push_back((uint16_t)term.size());
    }
    if (!std::equal(row.begin(), row.end(), C.begin() + (size_t)a * kd) || term.size() > 60000) return B;
  }
  B.mb = mb;
  B.index = index;
  B.term = term;
  return B;
}

}  // namespace mea
