// heget.cuh's FP32 vertex and current functions with every rounding written out.
//
// heget.cuh leaves it to the compiler which products and sums become one
// multiply-add, and its choice can change with the code around a call (a
// momentum loaded another way, a caller unrolled differently), which moves
// results by their rounding.  The kernel that uses these functions
// (amp_phased_kernel.cu) has to give the per-lane program's amplitudes bit for
// bit however it is arranged; so the choices the per-lane kernels get are
// fixed here: a complex product is (fma(ar, br, -(ai bi)), fma(ai, br, ar bi)) or,
// where one factor is a stored and the other a computed value,
// (.., fma(ar, bi, ai br)); sums of complex products are separate additions, real
// times complex plus a sum is a multiply-add.
#pragma once
#include "heget.cuh"

namespace mea {
namespace pinned {

typedef cx<float> C;
typedef W4<float> V;

__device__ __forceinline__ C mul(C a, C b) {
  return {__fmaf_rn(a.r, b.r, -__fmul_rn(a.i, b.i)), __fmaf_rn(a.i, b.r, __fmul_rn(a.r, b.i))};
}
// the same product with the other imaginary product rounded first
__device__ __forceinline__ C mul2(C a, C b) {
  return {__fmaf_rn(a.r, b.r, -__fmul_rn(a.i, b.i)), __fmaf_rn(a.r, b.i, __fmul_rn(a.i, b.r))};
}
__device__ __forceinline__ C add(C a, C b) { return {__fadd_rn(a.r, b.r), __fadd_rn(a.i, b.i)}; }
__device__ __forceinline__ C sub(C a, C b) { return {__fsub_rn(a.r, b.r), __fsub_rn(a.i, b.i)}; }
__device__ __forceinline__ C scale(float f, C a) { return {__fmul_rn(f, a.r), __fmul_rn(f, a.i)}; }
__device__ __forceinline__ C mac(float f, C a, C s) { return {__fmaf_rn(f, a.r, s.r), __fmaf_rn(f, a.i, s.i)}; }  // f a + s
__device__ __forceinline__ C neg(C a) { return {-a.r, -a.i}; }

// metric (or plain) product of two vectors
template <bool PLAIN = false>
__device__ __forceinline__ C dot(const V& a, const V& b) {
  C s = mul(a.c[0], b.c[0]);
#pragma unroll
  for (int k = 1; k < 4; ++k) s = PLAIN ? add(s, mul(a.c[k], b.c[k])) : sub(s, mul(a.c[k], b.c[k]));
  return s;
}
// a stored wavefunction with one that was just computed
template <bool PLAIN = false>
__device__ __forceinline__ C dot2(const V& a, const V& b) {
  C s = mul2(a.c[0], b.c[0]);
#pragma unroll
  for (int k = 1; k < 4; ++k) s = PLAIN ? add(s, mul2(a.c[k], b.c[k])) : sub(s, mul2(a.c[k], b.c[k]));
  return s;
}
__device__ __forceinline__ C dot(const float* p, const V& a) {
  C s = mac(p[0], a.c[0], neg(scale(p[1], a.c[1])));
  s = mac(-p[2], a.c[2], s);
  return mac(-p[3], a.c[3], s);
}

__device__ __forceinline__ V vvv_part(const V& y, const V& z, const float* k1, const float* k2, const float* k3, float g) {
  float d12[4], d23[4], d31[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    d12[m] = __fsub_rn(k1[m], k2[m]);
    d23[m] = __fsub_rn(k2[m], k3[m]);
    d31[m] = __fsub_rn(k3[m], k1[m]);
  }
  const C ay = scale(-g, dot(d12, z)), az = scale(-g, dot(d31, y)), ad = scale(-g, dot(y, z));
  V o;
#pragma unroll
  for (int m = 0; m < 4; ++m) o.c[m] = mac(d23[m], ad, add(mul(ay, y.c[m]), mul(az, z.c[m])));
  return o;
}
__device__ __forceinline__ C vvv_amp(const V& x, const V& y, const V& z, const float* kx, const float* ky, const float* kz,
                                     float g) {
  return dot2(x, vvv_part(y, z, kx, ky, kz, g));
}
__device__ __forceinline__ V jvv(const V& x, const V& y, const float* kx, const float* ky, float inv_q2, float g) {
  float k_open[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) k_open[m] = -__fadd_rn(kx[m], ky[m]);
  V o = vvv_part(x, y, k_open, kx, ky, g);
#pragma unroll
  for (int m = 0; m < 4; ++m) o.c[m] = scale(inv_q2, o.c[m]);
  return o;
}
__device__ __forceinline__ V gggg_part(const V& x, const V& y, const V& z, float gg) {
  const C xy = scale(gg, dot(x, y)), xz = scale(gg, dot(x, z));
  V o;
#pragma unroll
  for (int m = 0; m < 4; ++m) o.c[m] = sub(mul(xy, z.c[m]), mul(xz, y.c[m]));
  return o;
}
__device__ __forceinline__ C gggg_amp(const V& a, const V& b, const V& c, const V& d, float gg) {
  return dot(a, gggg_part(b, c, d, gg));
}
__device__ __forceinline__ V jggg(const V& a, const V& b, const V& c, float inv_q2, float gg) {
  V o = gggg_part(c, b, a, gg);
#pragma unroll
  for (int m = 0; m < 4; ++m) o.c[m] = scale(inv_q2, o.c[m]);
  return o;
}

// V0 +- V3, V1 -+ i V2
struct Slash {
  C p, m, x, y;  // plus, minus, V1 - i V2, V1 + i V2
  __device__ __forceinline__ explicit Slash(const V& v) {
    p = add(v.c[0], v.c[3]);
    m = sub(v.c[0], v.c[3]);
    const C iv = {-v.c[2].i, v.c[2].r};
    x = sub(v.c[1], iv);
    y = add(v.c[1], iv);
  }
};
__device__ __forceinline__ V slash_col(const V& v, const V& s) {
  const Slash l(v);
  V o;
  o.c[0] = sub(mul2(l.m, s.c[2]), mul(l.x, s.c[3]));
  o.c[1] = sub(mul2(l.p, s.c[3]), mul(l.y, s.c[2]));
  o.c[2] = add(mul2(l.p, s.c[0]), mul(l.x, s.c[1]));
  o.c[3] = add(mul(l.y, s.c[0]), mul2(l.m, s.c[1]));
  return o;
}
__device__ __forceinline__ V row_slash(const V& s, const V& v) {
  const Slash l(v);
  V o;
  o.c[0] = add(mul(s.c[2], l.p), mul2(s.c[3], l.y));
  o.c[1] = add(mul2(s.c[2], l.x), mul(s.c[3], l.m));
  o.c[2] = sub(mul(s.c[0], l.m), mul2(s.c[1], l.y));
  o.c[3] = sub(mul(s.c[1], l.p), mul2(s.c[0], l.x));
  return o;
}
// (px - i py) s and (px + i py) s
__device__ __forceinline__ C mul_m(float px, float py, C s) {
  return {__fmaf_rn(px, s.r, __fmul_rn(py, s.i)), __fmaf_rn(px, s.i, -__fmul_rn(py, s.r))};
}
__device__ __forceinline__ C mul_p(float px, float py, C s) {
  return {__fmaf_rn(px, s.r, -__fmul_rn(py, s.i)), __fmaf_rn(px, s.i, __fmul_rn(py, s.r))};
}
__device__ __forceinline__ V slash_real_col(const float* P, const V& s) {
  const float vp = __fadd_rn(P[0], P[3]), vm = __fsub_rn(P[0], P[3]);
  V o;
  o.c[0] = mac(vm, s.c[2], neg(mul_m(P[1], P[2], s.c[3])));
  o.c[1] = mac(vp, s.c[3], neg(mul_p(P[1], P[2], s.c[2])));
  o.c[2] = mac(vp, s.c[0], mul_m(P[1], P[2], s.c[1]));
  o.c[3] = mac(vm, s.c[1], mul_p(P[1], P[2], s.c[0]));
  return o;
}
__device__ __forceinline__ V row_slash_real(const V& s, const float* P) {
  const float vp = __fadd_rn(P[0], P[3]), vm = __fsub_rn(P[0], P[3]);
  V o;
  o.c[0] = mac(vp, s.c[2], mul_p(P[1], P[2], s.c[3]));
  o.c[1] = mac(vm, s.c[3], mul_m(P[1], P[2], s.c[2]));
  o.c[2] = mac(vm, s.c[0], neg(mul_p(P[1], P[2], s.c[1])));
  o.c[3] = mac(vp, s.c[1], neg(mul_m(P[1], P[2], s.c[0])));
  return o;
}
__device__ __forceinline__ V fvi(const V& fi, const V& v, const float* P, float inv_p2, float g) {
  V u = slash_real_col(P, slash_col(v, fi));
  const float f = __fmul_rn(-g, inv_p2);
#pragma unroll
  for (int m = 0; m < 4; ++m) u.c[m] = scale(f, u.c[m]);
  return u;
}
__device__ __forceinline__ V fvo(const V& fo, const V& v, const float* P, float inv_p2, float g) {
  V u = row_slash_real(row_slash(fo, v), P);
  const float f = __fmul_rn(g, inv_p2);
#pragma unroll
  for (int m = 0; m < 4; ++m) u.c[m] = scale(f, u.c[m]);
  return u;
}
// f fo gamma^mu fi
__device__ __forceinline__ V pair_current(const V& a, const V& b, float f) {
  const C p02 = mul2(a.c[0], b.c[2]), p13 = mul2(a.c[1], b.c[3]), p20 = mul2(a.c[2], b.c[0]), p31 = mul2(a.c[3], b.c[1]);
  const C p03 = mul2(a.c[0], b.c[3]), p12 = mul2(a.c[1], b.c[2]), p21 = mul2(a.c[2], b.c[1]), p30 = mul2(a.c[3], b.c[0]);
  const C t = sub(add(sub(p12, p03), p21), p30);
  V j;
  j.c[0] = scale(f, add(add(add(p02, p13), p20), p31));
  j.c[1] = scale(f, sub(sub(add(p03, p12), p21), p30));
  j.c[2] = scale(f, C{-t.i, t.r});
  j.c[3] = scale(f, add(sub(sub(p02, p13), p20), p31));
  return j;
}
__device__ __forceinline__ V jio(const V& fi, const V& fo, float inv_q2, float g) {
  return pair_current(fo, fi, __fmul_rn(-g, inv_q2));
}
__device__ __forceinline__ V iov_part_v(const V& fi, const V& fo, float g) { return pair_current(fo, fi, g); }
__device__ __forceinline__ V iov_part_i(const V& fo, const V& v, float g) {
  V t = row_slash(fo, v);
#pragma unroll
  for (int m = 0; m < 4; ++m) t.c[m] = scale(g, t.c[m]);
  return t;
}
__device__ __forceinline__ V iov_part_o(const V& fi, const V& v, float g) {
  V t = slash_col(v, fi);
#pragma unroll
  for (int m = 0; m < 4; ++m) t.c[m] = scale(g, t.c[m]);
  return t;
}
__device__ __forceinline__ C iov_amp(const V& fi, const V& fo, const V& v, float g) {
  return scale(g, dot2<true>(fo, slash_col(v, fi)));
}

}  // namespace pinned
}  // namespace mea
