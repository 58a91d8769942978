// Base of a process's colour amplitudes (see colour_base.h).
#include "colour_base.h"

#include <algorithm>

namespace mea {

typedef uint32_t u32;
typedef uint64_t u64;
static const u64 kPrime = 2147483647ull;  // 2^31 - 1: x mod it is a sum of 31-bit digits

static inline u32 reduce(u64 x) {  // x < 2^63
  x = (x & kPrime) + (x >> 31);
  x = (x & kPrime) + (x >> 31);
  return (u32)(x >= kPrime ? x - kPrime : x);
}
static u32 inverse(u32 a) {
  u64 r = 1, x = a;
  for (u64 e = kPrime - 2; e; e >>= 1, x = reduce(x * x))
    if (e & 1) r = reduce(r * x);
  return (u32)r;
}
// x += f y (mod the prime)
static void add_multiple(std::vector<u32>& x, u32 f, const std::vector<u32>& y, size_t n) {
  for (size_t j = 0; j < n; ++j) x[j] = reduce(x[j] + (u64)f * y[j]);
}

// Base of the rows of C (m x kd small integers): the first rows that no
// earlier ones generate, and the others as sums of them, by elimination
// modulo a prime on `cols` random combinations of the columns (checked exactly
// below).  Returns false unless the base is rows 0 .. mb - 1 and every
// coefficient is 0, 1 or -1.
static bool find_base(const std::vector<int>& C, int m, int kd, int cols, int& mb, std::vector<std::vector<int>>& coef) {
  u64 seed = 0x9E3779B97F4A7C15ull;
  std::vector<u32> rnd((size_t)kd * cols);
  for (u32& x : rnd) {  // a linear congruential sequence
    seed = seed * 6364136223846793005ull + 1442695040888963407ull;
    x = (u32)((seed >> 33) % kPrime);
  }
  std::vector<int64_t> sum((size_t)m * cols, 0);  // below kd max|c| 2^31
  for (int a = 0; a < m; ++a)
    for (int d = 0; d < kd; ++d) {
      const int64_t c = C[(size_t)a * kd + d];
      if (!c) continue;
      int64_t* s = &sum[(size_t)a * cols];
      const u32* x = &rnd[(size_t)d * cols];
      for (int j = 0; j < cols; ++j) s[j] += c * (int64_t)x[j];
    }
  std::vector<std::vector<u32>> B, T;  // reduced rows and what they are of the base rows
  std::vector<int> piv;
  mb = 0;
  coef.clear();
  for (int a = 0; a < m; ++a) {
    std::vector<u32> r(cols), c(m, 0);
    for (int j = 0; j < cols; ++j) r[j] = (u32)(((sum[(size_t)a * cols + j] % (int64_t)kPrime) + (int64_t)kPrime) % (int64_t)kPrime);
    for (size_t b = 0; b < B.size(); ++b) {
      const u32 f = r[piv[b]];
      if (!f) continue;
      add_multiple(r, (u32)kPrime - f, B[b], cols);
      add_multiple(c, f, T[b], mb);
    }
    int q = -1;
    for (int j = 0; j < cols && q < 0; ++j)
      if (r[j]) q = j;
    if (q >= 0) {
      if (a != mb) return false;  // the base is not a prefix
      const u32 iv = inverse(r[q]);
      for (u32& x : r) x = reduce((u64)x * iv);
      std::vector<u32> tb(m, 0);
      for (int j = 0; j < mb; ++j) tb[j] = reduce((u64)(c[j] ? (u32)kPrime - c[j] : 0) * iv);
      tb[mb] = iv;
      B.push_back(r);
      T.push_back(tb);
      piv.push_back(q);
      ++mb;
    } else {
      std::vector<int> k(m, 0);
      for (int j = 0; j < mb; ++j) {
        if (c[j] == 1) k[j] = 1;
        else if (c[j] == kPrime - 1) k[j] = -1;
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
  // The strings of one quark line are independent, those of two lines depend on
  // each other with other coefficients than 1 and -1: nothing to look for.
  if (p.family != FAM_GLUON) return B;
  // (n-2)! of the orderings are independent; that many random combinations and a few
  // more tell the rows apart (a larger rank would fail the exact check)
  int rank = 1;
  for (int k = 2; k <= p.n_ext - 2; ++k) rank *= k;
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
  if (!find_base(C, m, kd, std::min(m, rank) + 8, mb, coef) || mb >= m) return B;
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
