// FP32 filters in front of the exact FP64 decisions.
//
// GB300 retires 2 FP64 results per SM and cycle and 128 FP32 results, so the
// evaluation kernels were bound by FP64 arithmetic whose answer is a yes or
// no (a quality not above a bound, an edge longer than L_up, a point on one
// side of a line), most of which single precision with a rigorous error bound
// can give (a batch of 512 meshes: 445 -> 414 ms with the flip gains', 377 with the
// collapses', 323 with the smoothing's filters).  Every filter returns "undecided"
// unless its answer is certain for the value the FP64 code computes; the caller then
// runs that code.  So no result changes, only the number of FP64 instructions behind
// it.
//
// Input: one 32-byte record per vertex (one DRAM sector; position and metric
// in double take 48 bytes in two sectors): each coordinate as two floats
// xh = RN(x), xl = RN(x - xh), the metric rounded to float, and `e`, an
// absolute error that covers what two floats leave out.
//
// Error bounds, u = 2^-24 (half an ulp).  A coordinate is x = xh + xl + d,
// |d| <= u^2 |x|.  The difference D = (qh - ph) + (ql - pl): the first
// subtraction is exact when the operands are within a factor of two, else its
// rounding is relative to D; so
//   |D - (q - p)| <= 3 u |D| + e_q + e_p,   e = 2^-46 max(|x|, |y|) + 1e-37
// (twice the bound u |ql - pl| + u^2 (|q| + |p|)).  Everything below bounds the
// rounding of its own formula on top of that; constants are rounded up.  The
// FP64 code's own rounding error is that of the same formula with 2^-53 in
// place of u, far inside the margin.  Overflow and NaN make every test false
// (undecided); underflow is covered by the absolute terms 1e-36.
//
// Plain C++ apart from the markers, so that a host build can check the bounds
// against exact arithmetic.
#pragma once

#include <math.h>
#include <string.h>

#ifdef __CUDACC__
#define PM_HD __host__ __device__ __forceinline__
#else
#define PM_HD inline
#endif

namespace pm {

struct VF {
  float xh, xl, yh, yl;
  float m00, m01, m11, e;
};

constexpr float kU = 5.9604645e-8f;  // 2^-24
constexpr float kTiny = 1e-36f;

// sqrt and reciprocal to within 2 u relative on either side (the device's
// approximate instructions are specified to 2^-23; inputs here are normal or
// lead to an undecided result)
PM_HD float f_sqrt(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return sqrtf(x);
#endif
}
PM_HD float f_rcp(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}

// The power of two of a positive normal number (its exponent bits), and its reciprocal.
PM_HD float f_pow2(float x) {
#ifdef __CUDA_ARCH__
  return __int_as_float(__float_as_int(x) & 0x7f800000);
#else
  int b;
  memcpy(&b, &x, 4);
  b &= 0x7f800000;
  memcpy(&x, &b, 4);
  return x;
#endif
}
PM_HD float f_pow2_inv(float x) {
#ifdef __CUDA_ARCH__
  return __int_as_float(0x7f000000 - (__float_as_int(x) & 0x7f800000));
#else
  int b;
  memcpy(&b, &x, 4);
  b = 0x7f000000 - (b & 0x7f800000);
  memcpy(&x, &b, 4);
  return x;
#endif
}

// The record of a position without a metric (orientations only).
PM_HD VF make_vf_xy(double x, double y) {
  VF v;
  v.m00 = v.m01 = v.m11 = 0.0f;
  v.xh = (float)x;
  v.xl = (float)(x - (double)v.xh);
  v.yh = (float)y;
  v.yl = (float)(y - (double)v.yh);
  v.e = 1.4210855e-14f * fmaxf(fabsf(v.xh), fabsf(v.yh)) + 1e-37f;  // 2^-46
  return v;
}

PM_HD VF make_vf(double x, double y, double m00, double m01, double m11) {
  VF v = make_vf_xy(x, y);
  v.m00 = (float)m00;
  v.m01 = (float)m01;
  v.m11 = (float)m11;
  // a metric that single precision cannot hold with full relative precision:
  // every test of the vertex is undecided
  const bool holds = v.m00 > 1e-30f && v.m00 < 1e30f && v.m11 > 1e-30f && v.m11 < 1e30f;
  if (!holds) v.e = INFINITY;
  return v;
}

PM_HD float f_dx(const VF& p, const VF& q) { return (q.xh - p.xh) + (q.xl - p.xl); }
PM_HD float f_dy(const VF& p, const VF& q) { return (q.yh - p.yh) + (q.yl - p.yl); }

// Twice the signed area of (p, q, r) and a bound of its error.  Products of
// differences: 2 * 3 u + u each, their difference u: 8 u (|t1| + |t2|), taken
// as 10 u; the absolute parts E of the differences enter linearly and squared.
struct FDet {
  float det, err;
};
PM_HD FDet f_det(float ax, float ay, float bx, float by, float E) {
  const float t1 = ax * by, t2 = ay * bx;
  FDet d;
  d.det = t1 - t2;
  const float sum = (fabsf(ax) + fabsf(ay)) + (fabsf(bx) + fabsf(by));
  d.err = 10.0f * kU * (fabsf(t1) + fabsf(t2)) + (1.25f * E * (sum + 2.0f * E) + kTiny);
  return d;
}

// Sign of the exact orientation of (p, q, r): +1, -1, or 0 when undecided.
PM_HD int f_orient(const VF& p, const VF& q, const VF& r) {
  const FDet d = f_det(f_dx(p, q), f_dy(p, q), f_dx(p, r), f_dy(p, r), p.e + (q.e + r.e));
  return d.det > d.err ? 1 : (d.det < -d.err ? -1 : 0);
}

// Squared length of (dx, dy) under the metric (k00, k01, k11), relative error
// `ku` of its entries (of |k01|'s bound sqrt(k00 k11) for k01), and a bound of
// the error: (ku + 8 u) (t0 + |t1| + t2) for the three terms, 2 u of the same
// for their sum, and |t1| <= t0 + t2 for a positive definite metric.
struct FLen {
  float L2, err;
};
PM_HD FLen f_len2(float k00, float k01, float k11, float dx, float dy, float E, float ku) {
  const float t0 = (k00 * dx) * dx, t2 = (k11 * dy) * dy;
  FLen l;
  l.L2 = (t0 + ((2.0f * k01) * dx) * dy) + t2;
  l.err = (2.0f * ku + 24.0f * kU) * (t0 + t2) +
          (4.0f * E * (k00 + k11) * ((fabsf(dx) + fabsf(dy)) + E) + kTiny);
  return l;
}

// Squared metric length of edge (a, b) under the mean of its ends' metrics.
PM_HD FLen f_edge2(const VF& a, const VF& b) {
  return f_len2(0.5f * (a.m00 + b.m00), 0.5f * (a.m01 + b.m01), 0.5f * (a.m11 + b.m11),
                f_dx(a, b), f_dy(a, b), a.e + b.e, 2.0f * kU);
}

// The length against a bound t whose square lies between lo2 and hi2 (floats
// rounded outwards): +1 certainly longer, -1 certainly shorter, 0 undecided.
PM_HD int f_len_cmp(const FLen& l, float lo2, float hi2) {
  return l.L2 - l.err > hi2 ? 1 : (l.L2 + l.err < lo2 ? -1 : 0);
}

// Bounds of the quality (12 sqrt 3 A / P^2) F(P / 3) of element (a, b, c) in its
// mean metric: `up` is NaN and `lo` -1 when they would be loose, and `lo` is -1
// unless the element is certainly counter-clockwise.  The quality grows with the
// area and the metric's determinant, which are taken at their bounds; as a function of
// P it is h(P) = F(P / 3) / P^2 with |d ln h / d ln P| <= 5 (between -2 and 1 below the
// ideal perimeter, between -5 and -2 above), so a relative error rP of P changes it by
// at most 5 rP to first order (rP <= 0.04 is required, the rest of the series is inside
// the factor 1.15).  The determinant is taken of the metric divided by k00's power of
// two (exact): of the entries themselves the product k00 k11 leaves single precision at
// half the decades that a record holds, and a mesh in small or large units would get no
// bound.  `sign` receives the orientation's sign, 0 when undecided.  `kx`
// bounds the relative error of one vertex's metric beyond its rounding (see
// f_metric_at): it adds to that of the mean, and four times to the determinant's.
struct FQual {
  float lo, up;
};

PM_HD FQual f_quality(const VF& a, const VF& b, const VF& c, int& sign, float kx = 0.0f) {
  const float E = a.e + (b.e + c.e);
  const float dx0 = f_dx(a, b), dy0 = f_dy(a, b);
  const float dx1 = f_dx(b, c), dy1 = f_dy(b, c);
  const float dx2 = f_dx(a, c), dy2 = f_dy(a, c);
  const FDet d = f_det(dx0, dy0, dx2, dy2, E);
  sign = d.det > d.err ? 1 : (d.det < -d.err ? -1 : 0);
  constexpr float third = 0.33333334f;
  const float k00 = ((a.m00 + b.m00) + c.m00) * third;
  const float k01 = ((a.m01 + b.m01) + c.m01) * third;
  const float k11 = ((a.m11 + b.m11) + c.m11) * third;
  const float ku = 5.0f * kU + kx;
  const FLen q0 = f_len2(k00, k01, k11, dx0, dy0, E, ku);
  const FLen q1 = f_len2(k00, k01, k11, dx1, dy1, E, ku);
  const FLen q2 = f_len2(k00, k01, k11, dx2, dy2, E, ku);
  const float l0 = f_sqrt(q0.L2), l1 = f_sqrt(q1.L2), l2 = f_sqrt(q2.L2);
  const float P = (l0 + l1) + l2;
  const float rp = f_rcp(P);
  // sqrt(L2) - sqrt(L2 - err) <= 0.75 err / sqrt(L2) while err <= L2 / 2
  const float eP = 0.75f * ((q0.err * f_rcp(l0) + q1.err * f_rcp(l1)) + q2.err * f_rcp(l2));
  const float rP = eP * rp + 6.0f * kU;
  const float two = f_pow2(k00), inv = f_pow2_inv(k00);
  const float s00 = k00 * inv, s01 = k01 * inv, s11 = k11 * inv, kk = s00 * s11;
  // (perimeters and metrics whose powers would underflow give no bound)
  const bool fine = rP < 0.04f && kx < 0.05f && q0.err < 0.4f * q0.L2 && q1.err < 0.4f * q1.L2 &&
                    q2.err < 0.4f * q2.L2 && P > 1e-6f && P < 1e6f && kk > 1e-30f;
  const float D = kk - s01 * s01, eD = (28.0f * kU + 4.2f * kx) * kk;
  const float up = 0.5f * (d.det + d.err);
  const float area = up < 0.0f ? 0.0f : up;  // a negative quality is below 0 (a NaN stays)
  const float x = P * third;
  const float s = x > 1.0f ? 3.0f * rp : x;
  const float f = s * (2.0f - s);
  const float h = (rp * rp) * ((f * f) * f), eh = 5.75f * rP + 40.0f * kU;
  const float w = 20.784612f * two;
  const float q = ((w * area) * f_sqrt(D + eD)) * h;
  const float p = ((w * (0.5f * (d.det - d.err))) * f_sqrt(D - eD)) * h;
  FQual r;
  r.up = fine ? q + (q * eh + 1e-30f) : nanf("");
  r.lo = fine && sign > 0 && D > eD ? p - (p * eh + 1e-30f) : -1.0f;
  return r;
}

PM_HD float f_quality_up(const VF& a, const VF& b, const VF& c, int& sign, float kx = 0.0f) {
  return f_quality(a, b, c, sign, kx).up;
}

// The barycentric metric at point x of element (a, b, d), into the metric part of
// `out`; returns a bound of its relative error (of m01's bound sqrt(m00 m11) for
// m01), NaN when the element's area is not known well enough.  A weight s / o
// has the error (err_s + |s / o| err_o) / o and roundings; by Cauchy the error of
// m01 stays below the larger of those of m00 and m11.
PM_HD float f_metric_at(const VF& x, const VF& a, const VF& b, const VF& d, VF& out) {
  const float E = (x.e + a.e) + (b.e + d.e);
  const float abx = f_dx(a, b), aby = f_dy(a, b), adx = f_dx(a, d), ady = f_dy(a, d);
  const float axx = f_dx(a, x), axy = f_dy(a, x);
  const FDet o = f_det(abx, aby, adx, ady, E);
  const FDet s0 = f_det(f_dx(x, b), f_dy(x, b), f_dx(x, d), f_dy(x, d), E);
  const FDet s1 = f_det(axx, axy, adx, ady, E), s2 = f_det(abx, aby, axx, axy, E);
  const float r = f_rcp(o.det);
  const float l0 = s0.det * r, l1 = s1.det * r, l2 = s2.det * r;
  const float e0 = 1.4f * (s0.err + fabsf(l0) * o.err) * r + 6.0f * kU * fabsf(l0);
  const float e1 = 1.4f * (s1.err + fabsf(l1) * o.err) * r + 6.0f * kU * fabsf(l1);
  const float e2 = 1.4f * (s2.err + fabsf(l2) * o.err) * r + 6.0f * kU * fabsf(l2);
  out.m00 = (l0 * a.m00 + l1 * b.m00) + l2 * d.m00;
  out.m01 = (l0 * a.m01 + l1 * b.m01) + l2 * d.m01;
  out.m11 = (l0 * a.m11 + l1 * b.m11) + l2 * d.m11;
  const float w0 = e0 + 5.0f * kU * fabsf(l0), w1 = e1 + 5.0f * kU * fabsf(l1),
              w2 = e2 + 5.0f * kU * fabsf(l2);
  const float k0 = ((w0 * a.m00 + w1 * b.m00) + w2 * d.m00) * f_rcp(out.m00);
  const float k1 = ((w0 * a.m11 + w1 * b.m11) + w2 * d.m11) * f_rcp(out.m11);
  const bool fine = o.det > 4.0f * o.err && out.m00 > 0.0f && out.m11 > 0.0f;
  const float k = 1.1f * (k0 > k1 ? k0 : k1);
  return fine && k0 == k0 && k1 == k1 ? k : nanf("");
}

}  // namespace pm
