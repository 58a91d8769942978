// One item of an ordered-recursion stage (ordered.h) in FP64, shared by the
// kernel (ordered_kernel.cu) and its host check.
#pragma once
#include "heget.cuh"
#include "ordered.h"

namespace mea {

struct OrdEvent {
  double* area;        // this event's currents
  double* F;           // its amplitudes (re, im)
  const double* et;    // leg blocks of the event table
  const double* mt;    // mask rows: momentum, 1/P^2
  const int8_t* leg;   // [leg][4]: type, spinor kind, incoming
};

// two-component complex spinor
struct S2 {
  cx<double> a, b;
};

MEA_HD uint32_t ord_rev(uint32_t v, int nb) {
  uint32_t r = 0;
  for (int i = 0; i < nb; ++i) r |= (v >> i & 1u) << (nb - 1 - i);
  return r;
}
MEA_HD OrdRef ord_ref(const uint64_t* rec, int i) {
#ifdef __CUDA_ARCH__
  const unsigned long long v = __ldg(reinterpret_cast<const unsigned long long*>(rec) + i);
#else
  const unsigned long long v = rec[i];
#endif
  OrdRef r;
  r.off = (uint16_t)v;
  r.row = (uint8_t)(v >> 16);
  r.sh = (uint8_t)(v >> 24);
  r.nb = (uint8_t)(v >> 32);
  r.flags = (uint8_t)(v >> 40);
  r.pad = (uint16_t)(v >> 48);
  return r;
}
MEA_HD uint32_t ord_var(const OrdRef& r, uint32_t var) {
  uint32_t v = var >> r.sh & ((1u << r.nb) - 1u);
  return (r.flags & 1u) ? ord_rev(v, r.nb) : v;
}
MEA_HD W4<double> ord_ld(const double* p) {
  W4<double> w;
#ifdef __CUDA_ARCH__
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double2 u = reinterpret_cast<const double2*>(p)[k];
    w.c[k] = {u.x, u.y};
  }
#else
  for (int k = 0; k < 4; ++k) w.c[k] = {p[2 * k], p[2 * k + 1]};
#endif
  return w;
}
MEA_HD void ord_st(double* p, const W4<double>& w) {
#ifdef __CUDA_ARCH__
#pragma unroll
  for (int k = 0; k < 4; ++k) reinterpret_cast<double2*>(p)[k] = make_double2(w.c[k].r, w.c[k].i);
#else
  for (int k = 0; k < 4; ++k) { p[2 * k] = w.c[k].r; p[2 * k + 1] = w.c[k].i; }
#endif
}
MEA_HD W4<double> ord_gluon(const OrdEvent& E, const OrdRef& r, uint32_t var) {
  W4<double> w = ord_ld(E.area + 2 * (size_t)r.off + 8 * ord_var(r, var));
  if (r.flags & 2u)
    for (int k = 0; k < 4; ++k) w.c[k] = -w.c[k];
  return w;
}
MEA_HD S2 ord_spinor(const OrdEvent& E, const OrdRef& r, uint32_t var) {
  const double* p = E.area + 2 * (size_t)r.off + 4 * ord_var(r, var);
  return S2{{p[0], p[1]}, {p[2], p[3]}};
}
MEA_HD void ord_st(double* p, const S2& s) { p[0] = s.a.r; p[1] = s.a.i; p[2] = s.b.r; p[3] = s.b.i; }

// Multiply-adds are written out: the FP64 pipe takes one operation per product
// and sum otherwise (the compiler leaves a complex product's additions apart).
MEA_HD double ord_fma(double a, double b, double c) {
#ifdef __CUDA_ARCH__
  return fma(a, b, c);
#else
  return a * b + c;
#endif
}
// acc + a b and acc - a b
MEA_HD cx<double> ord_mac(cx<double> acc, cx<double> a, cx<double> b) {
  return {ord_fma(-a.i, b.i, ord_fma(a.r, b.r, acc.r)), ord_fma(a.i, b.r, ord_fma(a.r, b.i, acc.i))};
}
MEA_HD cx<double> ord_msc(cx<double> acc, cx<double> a, cx<double> b) {
  return {ord_fma(a.i, b.i, ord_fma(-a.r, b.r, acc.r)), ord_fma(-a.i, b.r, ord_fma(-a.r, b.i, acc.i))};
}
MEA_HD cx<double> ord_mul(cx<double> a, cx<double> b) {
  return {ord_fma(-a.i, b.i, a.r * b.r), ord_fma(a.i, b.r, a.r * b.i)};
}
MEA_HD cx<double> ord_macr(cx<double> acc, double a, cx<double> b) {
  return {ord_fma(a, b.r, acc.r), ord_fma(a, b.i, acc.i)};
}
MEA_HD cx<double> ord_dot(const W4<double>& a, const W4<double>& b) {
  return ord_msc(ord_msc(ord_msc(ord_mul(a.c[0], b.c[0]), a.c[1], b.c[1]), a.c[2], b.c[2]), a.c[3], b.c[3]);
}
MEA_HD cx<double> ord_dot(const double* p, const W4<double>& a) {
  cx<double> s = p[0] * a.c[0];
  for (int m = 1; m < 4; ++m) s = ord_macr(s, -p[m], a.c[m]);
  return s;
}
// acc += s x, acc -= s x
MEA_HD void ord_add(W4<double>& acc, cx<double> s, const W4<double>& x) {
  for (int m = 0; m < 4; ++m) acc.c[m] = ord_mac(acc.c[m], s, x.c[m]);
}
MEA_HD void ord_sub_from(W4<double>& acc, cx<double> s, const W4<double>& x) {
  for (int m = 0; m < 4; ++m) acc.c[m] = ord_msc(acc.c[m], s, x.c[m]);
}

// [a, b]; FULL false: conserved currents, Pa.a = Pb.b = 0 drops out
template <bool FULL>
MEA_HD void ord_bracket(W4<double>& acc, const W4<double>& a, const W4<double>& b, const double* pa, const double* pb) {
  cx<double> sb, sa;
  double d[4];
  for (int m = 0; m < 4; ++m) d[m] = pa[m] - pb[m];
  if (FULL) {
    double ca[4], cb[4];
    for (int m = 0; m < 4; ++m) {
      ca[m] = ord_fma(2.0, pb[m], pa[m]);
      cb[m] = ord_fma(2.0, pa[m], pb[m]);
    }
    sb = ord_dot(ca, a);
    sa = ord_dot(cb, b);
  } else {
    sb = 2.0 * ord_dot(pb, a);
    sa = 2.0 * ord_dot(pa, b);
  }
  const cx<double> ab = ord_dot(a, b);
  ord_add(acc, sb, b);
  ord_sub_from(acc, sa, a);
  for (int m = 0; m < 4; ++m) acc.c[m] = ord_macr(acc.c[m], d[m], ab);
}

// Sub-word i .. j (letters i .. j - 1) of a word of k letters in its record:
// row i of the triangular table, j = i + 1 .. k.
MEA_HD int ord_sub(int k, int i, int j) { return i * k - i * (i - 1) / 2 + (j - i - 1); }

// sum of [.,.] and {.,.,.} over the splits of the word whose pieces have at
// most `most` letters (longer ones are closed elsewhere)
template <bool FULL>
MEA_HD W4<double> ord_word_of(const OrdEvent& E, const uint64_t* rec, int k, uint32_t var, int most) {
  W4<double> acc;
  for (int m = 0; m < 4; ++m) acc.c[m] = {0.0, 0.0};
  for (int i = 1; i < k; ++i) {
    if (i > most || k - i > most) continue;
    const OrdRef ra = ord_ref(rec, ord_sub(k, 0, i)), rb = ord_ref(rec, ord_sub(k, i, k));
    ord_bracket<FULL>(acc, ord_gluon(E, ra, var), ord_gluon(E, rb, var), E.mt + 5 * ra.row, E.mt + 5 * rb.row);
  }
  for (int i = 1; i + 1 < k; ++i) {
    const W4<double> a = ord_gluon(E, ord_ref(rec, ord_sub(k, 0, i)), var);
    for (int j = i + 1; j < k; ++j) {
      const W4<double> b = ord_gluon(E, ord_ref(rec, ord_sub(k, i, j)), var);
      const W4<double> c = ord_gluon(E, ord_ref(rec, ord_sub(k, j, k)), var);
      const cx<double> ac = ord_dot(a, c), ab = ord_dot(a, b), bc = ord_dot(b, c);
      ord_add(acc, 2.0 * ac, b);
      ord_sub_from(acc, ab, c);
      ord_sub_from(acc, bc, a);
    }
  }
  return acc;
}
MEA_HD W4<double> ord_word(const OrdEvent& E, const uint64_t* rec, int k, uint32_t var, bool full, int most) {
  return full ? ord_word_of<true>(E, rec, k, var, most) : ord_word_of<false>(E, rec, k, var, most);
}

// acc + Jslash psi for a right-handed (components 2, 3 -> 0, 1) or left-handed (0, 1 -> 2, 3) column
MEA_HD S2 ord_slash(const S2& acc, const W4<double>& V, const S2& s, bool left) {
  const cx<double> vp = V.c[0] + V.c[3], vm = V.c[0] - V.c[3];
  const cx<double> m = V.c[1] - times_i(V.c[2]), p = V.c[1] + times_i(V.c[2]);
  if (left) return S2{ord_mac(ord_mac(acc.a, vp, s.a), m, s.b), ord_mac(ord_mac(acc.b, p, s.a), vm, s.b)};
  return S2{ord_msc(ord_mac(acc.a, vm, s.a), m, s.b), ord_msc(ord_mac(acc.b, vp, s.b), p, s.a)};
}
// acc + row psibar Jslash: right-handed row (components 0, 1 -> 2, 3) or left-handed (2, 3 -> 0, 1)
MEA_HD S2 ord_row_slash(const S2& acc, const S2& s, const W4<double>& V, bool left) {
  const cx<double> vp = V.c[0] + V.c[3], vm = V.c[0] - V.c[3];
  const cx<double> m = V.c[1] - times_i(V.c[2]), p = V.c[1] + times_i(V.c[2]);
  if (left) return S2{ord_mac(ord_mac(acc.a, s.a, vp), s.b, p), ord_mac(ord_mac(acc.b, s.a, m), s.b, vm)};
  return S2{ord_msc(ord_mac(acc.a, s.a, vm), s.b, p), ord_msc(ord_mac(acc.b, s.b, vp), s.a, m)};
}
// f times the same without acc for a real momentum
MEA_HD S2 ord_slash_real(const double* q, const S2& s, double f, bool left) {
  const double vp = f * (q[0] + q[3]), vm = f * (q[0] - q[3]), x = f * q[1], y = f * q[2];
  const cx<double> m = {x, -y}, p = {x, y};
  if (left) return S2{ord_mac(vp * s.a, m, s.b), ord_mac(vm * s.b, p, s.a)};
  return S2{ord_msc(vm * s.a, m, s.b), ord_msc(vp * s.b, p, s.a)};
}
MEA_HD S2 ord_row_slash_real(const S2& s, const double* q, double f, bool left) {
  const double vp = f * (q[0] + q[3]), vm = f * (q[0] - q[3]), x = f * q[1], y = f * q[2];
  const cx<double> m = {x, -y}, p = {x, y};
  if (left) return S2{ord_mac(vp * s.a, s.b, p), ord_mac(vm * s.b, s.a, m)};
  return S2{ord_msc(vm * s.a, s.b, p), ord_msc(vp * s.b, s.a, m)};
}
MEA_HD cx<double> ord_in(const S2& row, const S2& col) { return ord_mac(ord_mul(row.a, col.a), row.b, col.b); }

// row gamma^mu column of one chirality (heget.cuh jio without the propagator)
MEA_HD W4<double> ord_pair(const S2& r, const S2& c, bool left) {
  W4<double> j;
  const cx<double> p = ord_mul(r.a, c.a), q = ord_mul(r.b, c.b), u = ord_mul(r.a, c.b), v = ord_mul(r.b, c.a);
  j.c[0] = p + q;
  if (!left) {
    j.c[1] = u + v;
    j.c[2] = times_i(v - u);
    j.c[3] = p - q;
  } else {
    j.c[1] = -(u + v);
    j.c[2] = times_i(u - v);
    j.c[3] = q - p;
  }
  return j;
}

MEA_HD void ord_put(double* F, uint32_t i, cx<double> v, bool add) {
  if (add) { F[2 * i] += v.r; F[2 * i + 1] += v.i; }
  else { F[2 * i] = v.r; F[2 * i + 1] = v.i; }
}

// Item (word, pattern) of a stage.
//   EXT_G  rec 0: {off, leg, -, bits, fixed helicity bit}
//   EXT_Q  rec 0: {off, leg, -, -, flags: 1 row, 2 both chiralities}
//   G      rec 0: {off, row}; 1..: sub-words
//   GF     rec 0: {-, row, sh: closings}; sub-words; closings
//   GA     rec 0: {first F}; 1: eps of the root; 2..: sub-words
//   PSI    rec 0: {off, row, -, -, flags: 4 chirality is the pattern's top bit}; per split: gluon, spinor
//   BAR    the same with the row current first in word order
//   PF     as PSI with closings: rec 0 {sh: closings}, 1: row spinor, splits, closings {f, z = gluon letter}
//   X      rec 0: {off, row, flags: as PSI}; 1: row; 2: column
//   Z      rec 0: {off, row of x, row of the root}; 1: x; 2: eps of the root
//   PA     rec 0: {first F}; 1: row spinor; per split: gluon, spinor
MEA_HD void ord_item(const OrdStage& st, const uint64_t* rec, uint32_t var, const OrdEvent& E) {
  const OrdRef h = ord_ref(rec, 0);
  const int k = st.k;
  switch (st.type) {
    case ORD_EXT_G: {
      const int l = h.row;
      const double* o = E.et + 8 * l;
      const int lam = (h.nb ? var & 1u : (uint32_t)(h.flags & 1u)) ? 1 : -1;
      ord_st(E.area + 2 * (size_t)h.off + 8 * var, ext_gluon<double>(o, o + 3, lam, E.leg[4 * l + 2] == 0));
      break;
    }
    case ORD_EXT_Q: {
      const double* o = E.et + 8 * h.row;  // sqrt(2E), a, b
      const bool left = (h.flags & 2u) && (var & 1u);
      const double ra = o[0] * o[1];
      const cx<double> rb = {o[0] * o[2], o[0] * o[3]};
      S2 s = left ? S2{{-rb.r, rb.i}, {ra, 0.0}} : S2{{ra, 0.0}, rb};
      if (h.flags & 1u) s = S2{conj(s.a), conj(s.b)};
      ord_st(E.area + 2 * (size_t)h.off + 4 * var, s);
      break;
    }
    case ORD_G: {
      W4<double> w = ord_word(E, rec + 1, k, var, st.full != 0, k);
      const double inv = E.mt[5 * h.row + 4];
      for (int m = 0; m < 4; ++m) w.c[m] = inv * w.c[m];
      ord_st(E.area + 2 * (size_t)h.off + 8 * var, w);
      break;
    }
    case ORD_GF: {
      W4<double> w = ord_word(E, rec + 1, k, var, st.full != 0, k);
      const double inv = E.mt[5 * h.row + 4];
      for (int m = 0; m < 4; ++m) w.c[m] = inv * w.c[m];
      const uint64_t* cl = rec + 1 + k * (k + 1) / 2;
      for (int c = 0; c < h.sh; ++c) {
        const OrdRef q = ord_ref(cl, c);  // same layout as OrdClose
        const uint32_t f = q.off, z = (uint32_t)q.row | (uint32_t)q.sh << 8;
        const uint32_t xnb = q.nb, left = q.flags, rev = q.pad & 255u, neg = q.pad >> 8;
        const uint32_t vw = rev ? ord_rev(var, st.nb) : var;
        for (uint32_t x = 0; x < (1u << xnb); ++x) {
          const uint32_t va = left ? x << st.nb | vw : vw << xnb | x;
          for (uint32_t rb = 0; rb < (h.flags ? 2u : 1u); ++rb) {
            const uint32_t zi = h.flags ? 2 * x + rb : x;
            const cx<double> v = ord_dot(ord_ld(E.area + 2 * (size_t)z + 8 * zi), w);
            ord_put(E.F, f + (h.flags ? 2 * va + rb : va), neg ? -v : v, true);
          }
        }
      }
      break;
    }
    case ORD_GA: {
      const W4<double> w = ord_word(E, rec + 2, k, var, st.full != 0, k - 2);
      const OrdRef e = ord_ref(rec, 1);
      for (uint32_t rb = 0; rb < 2; ++rb)
        ord_put(E.F, h.off + 2 * var + rb, ord_dot(ord_ld(E.area + 2 * (size_t)e.off + 8 * rb), w), false);
      break;
    }
    case ORD_PSI:
    case ORD_BAR: {
      const bool left = (h.flags & 4u) && (var >> (st.nb - 1) & 1u);
      S2 t = {{0.0, 0.0}, {0.0, 0.0}};
      for (int i = 0; i < k; ++i) {
        const W4<double> g = ord_gluon(E, ord_ref(rec, 1 + 2 * i), var);
        const OrdRef rs = ord_ref(rec, 2 + 2 * i);
        // the spinor's bits: the line's chirality (top bit), then its letters
        const uint32_t sv = (h.flags & 4u) ? (var >> (st.nb - 1) << (rs.nb - 1) | (var >> rs.sh & ((1u << (rs.nb - 1)) - 1u)))
                                           : (var >> rs.sh & ((1u << rs.nb) - 1u));
        const double* p = E.area + 2 * (size_t)rs.off + 4 * sv;
        const S2 s = S2{{p[0], p[1]}, {p[2], p[3]}};
        t = st.type == ORD_PSI ? ord_slash(t, g, s, left) : ord_row_slash(t, s, g, left);
      }
      const double* q = E.mt + 5 * h.row;
      const S2 u = st.type == ORD_PSI ? ord_slash_real(q, t, q[4], !left) : ord_row_slash_real(t, q, -q[4], !left);
      ord_st(E.area + 2 * (size_t)h.off + 4 * var, u);
      break;
    }
    case ORD_PF: {
      S2 t = {{0.0, 0.0}, {0.0, 0.0}};
      for (int i = 0; i < k; ++i)
        t = ord_slash(t, ord_gluon(E, ord_ref(rec, 2 + 2 * i), var), ord_spinor(E, ord_ref(rec, 3 + 2 * i), var), false);
      const double* q = E.mt + 5 * h.row;
      const S2 u = ord_slash_real(q, t, q[4], true);
      const S2 row = ord_spinor(E, ord_ref(rec, 1), 0);
      const uint64_t* cl = rec + 2 + 2 * k;
      for (int c = 0; c < h.sh; ++c) {
        const OrdRef q2 = ord_ref(cl, c);
        const uint32_t f = q2.off, z = (uint32_t)q2.row | (uint32_t)q2.sh << 8, xnb = q2.nb;
        for (uint32_t x = 0; x < (1u << xnb); ++x)
          ord_put(E.F, f + (x << st.nb | var), ord_in(row, ord_slash(S2{{0.0, 0.0}, {0.0, 0.0}}, ord_ld(E.area + 2 * (size_t)z + 8 * x), u, false)), true);
      }
      break;
    }
    case ORD_X: {
      const bool left = (h.flags & 4u) && (var >> (st.nb - 1) & 1u);
      const OrdRef rr = ord_ref(rec, 1), rc = ord_ref(rec, 2);
      // row: chirality and its letters (high bits), column: chirality and its letters (low bits)
      const uint32_t top = var >> (st.nb - 1);
      const uint32_t vr = top << (rr.nb - 1) | (var >> rr.sh & ((1u << (rr.nb - 1)) - 1u));
      const uint32_t vc = top << (rc.nb - 1) | (var & ((1u << (rc.nb - 1)) - 1u));
      const double* pr = E.area + 2 * (size_t)rr.off + 4 * vr;
      const double* pc = E.area + 2 * (size_t)rc.off + 4 * vc;
      W4<double> j = ord_pair(S2{{pr[0], pr[1]}, {pr[2], pr[3]}}, S2{{pc[0], pc[1]}, {pc[2], pc[3]}}, left);
      const double inv = E.mt[5 * h.row + 4];
      for (int m = 0; m < 4; ++m) j.c[m] = inv * j.c[m];
      ord_st(E.area + 2 * (size_t)h.off + 8 * var, j);
      break;
    }
    case ORD_Z: {
      const OrdRef x = ord_ref(rec, 1), e = ord_ref(rec, 2);
      if (h.flags & 1u) {  // the current of the quark pair itself
        const S2 r = ord_spinor(E, x, 0), c = ord_spinor(E, e, 0);
        ord_st(E.area + 2 * (size_t)h.off, ord_pair(r, c, false));
      } else {
        W4<double> z;
        for (int m = 0; m < 4; ++m) z.c[m] = {0.0, 0.0};
        ord_bracket<false>(z, ord_ld(E.area + 2 * (size_t)x.off + 8 * (var >> 1)), ord_ld(E.area + 2 * (size_t)e.off + 8 * (var & 1u)),
                    E.mt + 5 * x.row, E.mt + 5 * e.row);
        ord_st(E.area + 2 * (size_t)h.off + 8 * var, z);
      }
      break;
    }
    default: {  // ORD_PA
      S2 t = {{0.0, 0.0}, {0.0, 0.0}};
      const int splits = h.sh;
      for (int i = 0; i < splits; ++i)
        t = ord_slash(t, ord_gluon(E, ord_ref(rec, 2 + 2 * i), var), ord_spinor(E, ord_ref(rec, 3 + 2 * i), var), false);
      ord_put(E.F, h.off + var, ord_in(ord_spinor(E, ord_ref(rec, 1), 0), t), false);
      break;
    }
  }
}

}  // namespace mea
