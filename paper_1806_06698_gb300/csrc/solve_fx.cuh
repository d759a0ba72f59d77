// solve_fx.cuh -- FP64 eigenpairs from an FP32 solve, refined in 62-bit fixed
// point on the integer pipes.
//
// GB300 executes 1.68 FP64 lanes per clock per SM but 64 lanes of the 32 x 32
// -> 64 bit product and of a 64-bit addition (measured), so a fixed-point
// multiply-add on 31-bit limbs (three products) costs a tenth of an FP64 one.
// Packed doubles of similar size are held in fixed point with 62 fractional
// bits; the eigenvalues' errors, about 2^-57 of the largest entry, are a tenth of
// FP64 rounding.  A matrix whose entries are all within 2^20 of the largest is
// solved so:
//   1. the method of C. F. Borges (arXiv 1806.06698, Secs. 1-1.4.1) in FP32
//      gives an approximate eigenvector frame, kept as a quaternion: R(q) is
//      a rotation whatever the rounding of q, so no orthogonalisation follows;
//   2. B = R^T A R in fixed point; the rotation that diagonalises it -- an
//      exact Jacobi rotation (Golub and Van Loan, Matrix Computations, 8.5)
//      of the closest pair, first-order perturbation towards the third -- is
//      formed in FP32 and multiplied into q, now with 30-bit components;
//   3. B is formed again from the new q.  |q|^2 is within 2^-27 of 1 (checked:
//      an integer quaternion of that length gives a rotation whatever steps
//      led to it) and B's off-diagonal entries are below
//      2^-27 (checked), so its diagonal holds the eigenvalues, and first-order
//      perturbation gives the eigenvectors: R (I + W + W^2/2), orthogonal to
//      rounding, W_ij = B_ij/(B_jj - B_ii) (Kato, Perturbation Theory for
//      Linear Operators, ch. 2).
// A matrix that fails the entry check or one of step 3 (graded or
// structured entries, three close eigenvalues, FP32 roots that did not
// converge) is left to the FP64 path.  The decision depends on the matrix
// alone, never on its neighbours in the batch, and every FP32 sum of products
// is an explicit fused operation, so that all builds of the kernels return
// the same bits.
#pragma once

#include <cstdint>

#include "arith.cuh"
#include "solve_f32.cuh"

namespace syev3 {
namespace fx {
namespace {  // internal linkage: every translation unit gets its own copy

// Fixed-point scales, in fractional bits: matrix entries (of A/2 after the
// pre-scale: |a/2| < 1/2) 62, rotation entries 60, A R and R^T A R 61.
// A number is split into a signed upper and a non-negative lower limb,
// v = h 2^31 + l (both with the sign of a for a matrix entry).  In a 3-term
// sum of products the h h and the h l + l h parts accumulate in one 64-bit
// register each; with the scales above neither overflows
// (|sum h l + l h| < 2^31 (sum |h_a| + sum |h_b|) <= 3.9 x 2^61), and l l is
// dropped, or replaced by its mean where that is not zero, through the
// accumulator's start.
struct Split {
  int h, l;
};

__device__ __forceinline__ Split split31(const int64_t v) { return {(int)(v >> 31), (int)v & 0x7fffffff}; }

// a b + c in one instruction (the plain expression was measured to become a
// product and a separate 64-bit addition in places).
__device__ __forceinline__ int64_t madw(const int a, const int b, const int64_t c) {
  int64_t d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

__device__ __forceinline__ void dot3(const Split a0, const Split a1, const Split a2, const Split b0, const Split b1,
                                     const Split b2, int64_t& hh, int64_t& cross) {
  hh = madw(a2.h, b2.h, madw(a1.h, b1.h, (int64_t)a0.h * b0.h));
  cross = madw(a0.h, b0.l, madw(a0.l, b0.h, cross));
  cross = madw(a1.h, b1.l, madw(a1.l, b1.h, cross));
  cross = madw(a2.h, b2.l, madw(a2.l, b2.h, cross));
}

// int64 -> float within 2^-23 relative: signed halves v = h 2^32 + l.
__device__ __forceinline__ float to_float(const int64_t v) {
  const int l = (int)v, h = (int)(v >> 32) + (int)((unsigned)l >> 31);
  return fmaf((float)h, 0x1p32f, (float)l);
}

// v 2^-frac as a double, rounded once: the halves become exact doubles by
// placing them in the fraction of a constant, so that two additions suffice.
template <int kFrac>
__device__ __forceinline__ double to_double(const int64_t v) {
  // upper half: 2^a + x 2^(32-frac), x = upper word + 2^31; lower: 2^b + lo 2^-frac
  constexpr int kHi = 1023 + 52 + 32 - kFrac, kLo = 1023 + 52 - kFrac;
  const double dh = __hiloint2double(kHi << 20, (int)((unsigned)(v >> 32) ^ 0x80000000u));
  const double dl = __hiloint2double(kLo << 20, (int)v);
  constexpr double u = 1.0 / (double)(1ull << (kFrac - 32));  // 2^(32-frac)
  constexpr double off = 0x1p52 * u + 0x1p31 * u + 0x1p20 * u;
  return (dh - off) + dl;
}

// v 2^(e-frac) as a double on the integer pipes, |v| < 2^63: normalised, rounded
// to nearest with ties away (v carries rounding errors of its own), the
// exponent added.  A zero upper word of |v| takes the form above, a result
// out of the normal range the general scaling; both rare.
template <int kFrac>
__device__ __forceinline__ double to_double_int(const int64_t v, const int e = 0) {
  const int64_t s = v >> 63;
  const uint64_t m = (uint64_t)((v ^ s) - s);
  const unsigned hi = (unsigned)(m >> 32), lo = (unsigned)m;
  if (hi == 0u) return mul_pow2(to_double<kFrac>(v), e);
  const int z = __clz((int)hi);
  const unsigned mh = __funnelshift_l(lo, hi, z), ml = lo << z;
  const uint64_t f = (((uint64_t)mh << 32 | ml) >> 11) + ((ml >> 10) & 1u);  // 53 bits, rounded
  const int E = 1023 + 62 - kFrac - z;  // exponent field at e = 0, less the leading bit's carry
  const int sign = (int)(s << 31);
  if ((unsigned)(E + e) > 2044u)
    return mul_pow2(__hiloint2double(((int)(f >> 32) + (E << 20)) | sign, (int)f), e);
  return __hiloint2double(((int)(f >> 32) + ((E + e) << 20)) | sign, (int)f);
}

// Rotation entries x 2^60 from an integer quaternion q with |q|^2 = 2^60
// (1 + eta): the numerators of R(q), row by row; norm receives |q|^2.
struct Quat {
  int w, x, y, z;
};

__device__ __forceinline__ void rotation(const Quat q, int64_t R[9], int64_t& norm) {
  const int64_t ww = (int64_t)q.w * q.w, xx = (int64_t)q.x * q.x, yy = (int64_t)q.y * q.y, zz = (int64_t)q.z * q.z;
  const int64_t s = ww - zz, d = xx - yy, p = ww + zz, e = xx + yy;
  norm = p + e;
  R[0] = s + d;
  R[4] = s - d;
  R[8] = p - e;
  const int64_t xy = (int64_t)q.x * q.y, xz = (int64_t)q.x * q.z, yz = (int64_t)q.y * q.z;
  const int w2 = 2 * q.w;
  R[1] = 2 * xy - (int64_t)w2 * q.z;
  R[3] = madw(w2, q.z, 2 * xy);
  R[2] = madw(w2, q.y, 2 * xz);
  R[6] = 2 * xz - (int64_t)w2 * q.y;
  R[5] = 2 * yz - (int64_t)w2 * q.x;
  R[7] = madw(w2, q.x, 2 * yz);
}

// (A/2) b for a column b of R, x 2^61.
__device__ __forceinline__ void times_column(const Split a[6], const Split b0, const Split b1, const Split b2,
                                             Split t[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const Split a0 = i == 0 ? a[0] : (i == 1 ? a[3] : a[4]);
    const Split a1 = i == 0 ? a[3] : (i == 1 ? a[1] : a[5]);
    const Split a2 = i == 0 ? a[4] : (i == 1 ? a[5] : a[2]);
    int64_t hh, cross = 1ll << 29;  // half a unit (the l l terms' signs are those of a)
    dot3(a0, a1, a2, b0, b1, b2, hh, cross);
    t[i] = split31((hh << 1) + (cross >> 30));
  }
}

__device__ __forceinline__ int64_t dot_column(const Split r0, const Split r1, const Split r2, const Split t[3]) {
  int64_t hh, cross = 0x70000000ll;  // mean of the l l terms (3 x 2^29) and half a unit
  dot3(t[0], t[1], t[2], r0, r1, r2, hh, cross);
  return (hh << 2) + (cross >> 29);
}

// R^T (A/2) R x 2^61 (upper triangle 00 01 11 02 12 22); a holds the limbs of
// the packed A/2 (11, 22, 33, 12, 13, 23) x 2^62, r those of R, 1 + eta times a
// rotation (norm = 2^60 (1 + eta)); trace: that of A/2 x 2^61.  The third diagonal entry is the trace's remainder -- R^T A R has the
// trace (1 + eta)^2 tr A -- so that only two of A R's columns are formed: 11
// products of three terms instead of 15.
__device__ __forceinline__ void rotated(const Split a[6], const Split r[9], const int64_t trace, const int64_t norm,
                                        int64_t B[6]) {
  Split t[3];
  times_column(a, r[0], r[3], r[6], t);
  B[0] = dot_column(r[0], r[3], r[6], t);
  B[3] = dot_column(r[2], r[5], r[8], t);
  times_column(a, r[1], r[4], r[7], t);
  B[1] = dot_column(r[0], r[3], r[6], t);
  B[2] = dot_column(r[1], r[4], r[7], t);
  B[4] = dot_column(r[2], r[5], r[8], t);
  const int64_t eta = norm - (1ll << 60);  // below 2^40
  const float etaf = to_float(eta);
  const int64_t both = 2 * eta + (int64_t)__float2int_rn(etaf * etaf * 0x1p-60f);  // (1 + eta)^2 - 1, x 2^60
  const Split T = split31(trace), E = split31(both);
  const int64_t grow = ((int64_t)T.h * E.h << 2) + (madw(T.h, E.l, (int64_t)T.l * E.h) >> 29);
  B[5] = trace + grow - B[0] - B[2];
}

// The power of two that brings v's largest component to [1/2, 1).
__device__ __forceinline__ float largest_to_half(const float v[3]) {
  int E = 1;
#pragma unroll
  for (int i = 0; i < 3; ++i) E = max(E, (__float_as_int(v[i]) >> 23) & 0xff);
  return pow2f(126 - E);
}

// The eigenvector frame of a (|a| < 1) by the FP32 method: outer
// eigenvectors u1 and u3 by their closed forms (or the deflated 2x2 solve),
// the third axis as their cross product; returned as an unnormalised
// quaternion with |q| in [2, 4].
struct QuatF {
  float w, x, y, z;
};

__device__ __forceinline__ QuatF frame32(const float a[6]) {
  using namespace f32;
  const Rot32 J = ordered_rotation32(a[0], a[3], a[1]);
  const float a1 = J.l1, a2 = J.l2, g = a[2];
  const float b1 = fmaf(J.c, a[4], J.s * a[5]), b2 = fmaf(J.c, a[5], -J.s * a[4]);
  const float ab = a1 - a2, bb1 = b1 * b1, bb2 = b2 * b2, h2 = fmaf(b1, b1, bb2);
  float v[3], u[3];
  // Sec. 1.1: deflated; also when a spike is so small that its square could
  // underflow (the test's right-hand side is 0 for a trace-free block).
  if (fabsf(ab * b1 * b2) <= 0x1p-23f * fabsf(a1 + a2) * h2 || fminf(fabsf(b1), fabsf(b2)) < 0x1p-60f) {
    const float rh = h2 > 0.f ? rsqrt32(h2) : 0.f, h = h2 * rh;
    const float gs = b1 * rh, gc = h2 > 0.f ? b2 * rh : 1.f;
    const Rot32 K = ordered_rotation32(fmaf(a1 * gs, gs, a2 * gc * gc), h, g);
    v[0] = gc; v[1] = -gs; v[2] = 0.f;
    u[0] = -gs * K.s; u[1] = -gc * K.s; u[2] = K.c;
  } else {
    float x[2];
    bool more[2];
    const P2 rab = pp(rcp32(ab)), b1p = make_float2(bb1, bb2), b2p = make_float2(bb2, bb1);
    const P2 g2 = psub(make_float2(g, a2), make_float2(a1, g));
    const P2 c = pmul(b2p, rab);
    roots32x2(pp(ab), rab, b1p, b2p, g2, c, psub(make_float2(-g2.x, -g2.y), c), x, more);
    const float mpa = x[0] + ab, npa = x[1] + ab;
    v[0] = b1 * mpa; v[1] = b2 * x[0]; v[2] = x[0] * mpa;
    u[0] = b1 * x[1]; u[1] = b2 * npa; u[2] = -(x[1] * npa);
    float vv = fmaf(v[0], v[0], fmaf(v[1], v[1], v[2] * v[2]));
    float uu = fmaf(u[0], u[0], fmaf(u[1], u[1], u[2] * u[2]));
    if (!(fminf(vv, uu) >= 0x1p-100f)) {  // squares near underflow (a small spike and a small abar beside g)
      const float sv = largest_to_half(v), su = largest_to_half(u);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        v[i] *= sv;
        u[i] *= su;
      }
      vv = fmaf(v[0], v[0], fmaf(v[1], v[1], v[2] * v[2]));
      uu = fmaf(u[0], u[0], fmaf(u[1], u[1], u[2] * u[2]));
    }
    const float iv = rsqrt32(vv), iu = rsqrt32(uu);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      v[i] *= iv;
      u[i] *= iu;
    }
  }
  // Columns v, u x v, u of the frame in the input's axes.
  const float r00 = fmaf(J.c, v[0], -J.s * v[1]), r10 = fmaf(J.s, v[0], J.c * v[1]), r20 = v[2];
  const float r02 = fmaf(J.c, u[0], -J.s * u[1]), r12 = fmaf(J.s, u[0], J.c * u[1]), r22 = u[2];
  const float r01 = fmaf(r12, r20, -r22 * r10), r11 = fmaf(r22, r00, -r02 * r20), r21 = fmaf(r02, r10, -r12 * r00);
  // 4 q_m q for the largest component q_m of the unit quaternion, read off
  // the rotation matrix (Shepperd 1978).
  const float ax = r21 - r12, ay = r02 - r20, az = r10 - r01, sxy = r01 + r10, sxz = r02 + r20, syz = r12 + r21;
  const bool neg = r22 < 0.f, s = neg ? r00 > r11 : r00 < -r11;
  const float d0 = neg ? 1.f - r22 : 1.f + r22, d1 = neg ? r00 - r11 : r00 + r11;
  const float t = s == neg ? d0 + d1 : d0 - d1;  // x and w cases add, y and z subtract
  QuatF q;
  if (neg) {
    q.w = s ? ax : ay;
    q.x = s ? t : sxy;
    q.y = s ? sxy : t;
    q.z = s ? sxz : syz;
  } else {
    q.w = s ? az : t;
    q.x = s ? sxz : ax;
    q.y = s ? syz : ay;
    q.z = s ? t : az;
  }
  return q;
}

// Step 2's rotation for B = (00 01 11 02 12 22): the closest pair (i, j) by a
// Jacobi rotation about the third axis k with the couplings to k eliminated
// to second order, then both towards k to first order; (i, j, k) cyclic.
// p receives the vector part x 2^30 of the quaternion (1; p).  Only ratios of B
// enter, so its scale is free.  False for a rotation towards k by more than
// about a radian, where first order says nothing; |p| <= 1 otherwise.
__device__ __forceinline__ bool small_rotation(const int64_t B[6], int p[3]) {
  const float e01 = to_float(B[1]), e02 = to_float(B[3]), e12 = to_float(B[4]);
  const float g01 = to_float(B[2] - B[0]), g12 = to_float(B[5] - B[2]), g02 = to_float(B[5] - B[0]);
  const float m01 = fabsf(g01), m12 = fabsf(g12), m02 = fabsf(g02);
  const bool k2 = m01 <= m12 && m01 <= m02, k0 = !k2 && m12 <= m02;  // else k = 1
  const float e = k2 ? e01 : (k0 ? e12 : e02), g = k2 ? g01 : (k0 ? g12 : -g02);
  const float fi = k2 ? e02 : (k0 ? e01 : e12), fj = k2 ? e12 : (k0 ? e02 : e01);
  const float ri = rcp32(k2 ? -g02 : (k0 ? g01 : g12)), rj = rcp32(k2 ? -g12 : (k0 ? g02 : -g01));
  const float wi = fi * ri, wj = fj * rj;
  const float ee = fmaf(0.5f, fmaf(fi, wj, fj * wi), e), gg = g + fmaf(fj, wj, -fi * wi);
  const float den = fabsf(gg) + sqrt32(fmaf(gg, gg, 4.f * ee * ee));
  float t = den > 0.f ? -2.f * ee * rcp32(den) : 0.f;
  t = gg < 0.f ? -t : t;
  const float h = t * rcp32(1.f + sqrt32(fmaf(t, t, 1.f)));  // tan of half the angle
  const float r = rcp32(fmaf(h, h, 1.f)), c = fmaf(2.f, r, -1.f), s = 2.f * h * r;
  const float oi = fmaf(c, fj, -s * fi) * rj, oj = -fmaf(c, fi, s * fj) * ri;
  const float wpi = fmaf(-h, oj, oi), wpj = fmaf(h, oi, oj);
  const int pi = __float2int_rn(0x1p29f * wpi), pj = __float2int_rn(0x1p29f * wpj);
  const int pk = __float2int_rn(0x1p30f * h);  // h below 0.42
  p[0] = k2 ? pi : (k0 ? pk : pj);
  p[1] = k2 ? pj : (k0 ? pi : pk);
  p[2] = k2 ? pk : (k0 ? pj : pi);
  return fmaxf(fabsf(wpi), fabsf(wpj)) <= 1.f;
}

// q (1; p), the components x 2^30 (|p| <= 1: the result is below 2^31).
__device__ __forceinline__ Quat times(const Quat q, const int p[3]) {
  constexpr int64_t half = 1ll << 29;
  Quat o;
  o.w = q.w - (int)(madw(q.z, p[2], madw(q.y, p[1], madw(q.x, p[0], half))) >> 30);
  o.x = q.x + (int)(madw(-q.z, p[1], madw(q.y, p[2], madw(q.w, p[0], half))) >> 30);
  o.y = q.y + (int)(madw(-q.x, p[2], madw(q.z, p[0], madw(q.w, p[1], half))) >> 30);
  o.z = q.z + (int)(madw(-q.y, p[0], madw(q.x, p[1], madw(q.w, p[2], half))) >> 30);
  return o;
}

// q scaled to |q|^2 = 2^60 (1 + eta), |eta| < 2^-27: an FP32 inverse square
// root with one Newton correction of the residual N s^2 - 1 (from 32-bit
// limbs, to 2^-30).
__device__ __forceinline__ Quat normalised(const Quat q) {
  const int64_t N = madw(q.z, q.z, madw(q.y, q.y, madw(q.x, q.x, (int64_t)q.w * q.w)));  // [2^59, 2^61)
  const int n31 = (int)(N >> 31);                     // N / 2^60 x 2^29
  const float s = rsqrt32((float)n31 * 0x1p-29f);     // (1/2, sqrt 2]
  const int si = __float2int_rn(s * 0x1p30f);         // exact
  const int s2 = (int)(((int64_t)si * si) >> 31);     // s^2 x 2^29
  const int res = (int)(((int64_t)n31 * s2 - (1ll << 58)) >> 27);  // (N s^2 - 1) x 2^31
  const int sc = si - (int)(((int64_t)si * res) >> 32);            // s (1 - res/2) x 2^30
  constexpr int64_t half = 1ll << 29;
  Quat o;
  o.w = (int)(madw(q.w, sc, half) >> 30);
  o.x = (int)(madw(q.x, sc, half) >> 30);
  o.y = (int)(madw(q.y, sc, half) >> 30);
  o.z = (int)(madw(q.z, sc, half) >> 30);
  return o;
}

// Largest |eta|, |q|^2 = 2^60 (1 + eta): what `rotated` and `solve` assume.
// Rounding leaves 2^-28 and seldom more.  A frame that came out NaN is q = 0 in integers:
// then B's off-diagonal entries are at rounding level too, and only this check
// refuses it.
constexpr int64_t kNormMax = (1ll << 33) - 4;
// Largest off-diagonal entry of the second B, 2^-27 (x 2^61); the rounding of
// q to 30 bits leaves up to 2^-28.
constexpr float kOffMax = 0x1p34f;
// Largest first-order rotation: W is held x 2^53 in 31 bits.
constexpr float kRotMax = 0x1p-23f;
// Largest second-order change of an eigenvalue, w e, 2^-56 (x 2^61): the same
// bound keeps the vectors' second-order terms below 2^-56 over their gap.
constexpr float kSecond = 0x1p5f;
// Off-diagonal entries at the rounding level of B (up to 2^-56) between values
// that are equal to that level: any vectors of the pair's plane will do.
constexpr float kNoise = 0x1p5f;

// e / g with the reciprocal's 2^-23 corrected by one Newton step.
__device__ __forceinline__ float quotient(const float e, const float g) {
  const float r = rcp32(g);
  return e * fmaf(r, fmaf(-g, r, 1.f), r);
}

// The packed matrix A as limbs of A 2^-e/2, its largest entry in [1/4, 1/2),
// when every off-diagonal entry is within 2^20 of the largest entry's exponent
// and every diagonal one is so or zero (similar), or there is no off-diagonal
// entry at all (diagonal); neither for a non-finite entry.  Entries within
// 2^8 are held exactly, smaller ones to 2^-62.
//
// The eigenvalues carry an error of about 2^-57 of the largest entry (rms; 2^-54
// at most), the vectors one of 2^-58 over the gap, whatever the eigenvalue's size.
// FP64 arithmetic loses 2^-53, but of the entries that an eigenvalue belongs to:
// it is the better one for graded matrices (D S D, D diagonal) with small rows.
// With kGraded (results in FP64) therefore
//  * a row or a 2x2 block below 2^-8 of the largest entry, or below 2^-6 beside an
//    entry that is not within 2^12, leaves the matrix to the FP64 path;
//  * so do a block below 2^-6 and two eigenvalues below 2^-6, for the vectors of
//    the pair;
//  * with a row below 2^-6, an eigenvalue below 2^-6 is formed again from its
//    vector and the record without rounding (small_value).
// Against double-double in a CPU build, relative error of the worst eigenvalue
// (median) and error of the worst vector (99 %), FP64 path / fixed point without
// this / with it: (1, d, d) with couplings d = 2^-12 4.9e-16, 3.1e-14, 4.9e-16 and
// 3e-16, 1e-14, 3e-16; D S D with D = (1, 1, 2^-5) 1.5e-16, 4.9e-15, below 1e-16;
// (1, 2^-5, 2^-5) 1.5e-16, 7.1e-15, 1.5e-16 and 7e-16, 1e-13, 7e-16; random D over
// 2^-6 1.7e-16, 3.1e-16, 1.4e-16 and 4e-16, 4e-15, 4e-16; ungraded gaussian entries
// 2.1e-16, below 1e-16 twice.  What remains: vectors of a pair at 2^-6 (D = (1,
// 2^-3, 2^-3)) 4e-15 at 99 %, the FP64 path 7e-16.  The lines are drawn where the
// fixed-point errors begin to exceed the other's and so that few generic matrices
// cross them: of well-separated spectra 6e-5 are formed again and 2e-5 more go to
// the FP64 path, whose serial chain adds 8 us to a small batch (leaving every
// entry spread beyond 2^8 to it: 2 %).  2^22 matrices, us: well-separated 439 ->
// 452, mixed 487 -> 503, tensors 440 -> 443, rank two 444 -> 597; eigenvalues only
// 340 -> 362, 374 -> 394, 340 -> 354, 344 -> 537; entries spread over 2^30, most of
// which the FP64 path takes again, 1273 -> 1636 (1570 when it took all).
constexpr unsigned kSpread = 20;
constexpr unsigned kWide = 12, kGraded6 = 6, kGraded8 = 8;
constexpr int64_t kSmall = 1ll << 54;  // eigenvalues x 2^60

struct Fixed {
  Split a[6];
  int e;
  bool similar, diagonal, finite;
  int graded;  // bit 0: a row below 2^-6 of the largest entry; bit 1: a 2x2 block
};

template <bool kGraded>
__device__ __forceinline__ Fixed fixed_of(const double a_in[6]) {
  Fixed F;
  unsigned h[6], l[6], top = 0u;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    h[i] = (unsigned)__double2hiint(a_in[i]);
    l[i] = (unsigned)__double2loint(a_in[i]);
    top = max(top, h[i] & 0x7fffffffu);
  }
  F.finite = top < 0x7ff00000u;
  F.diagonal = (((h[3] | h[4] | h[5]) << 1) | l[3] | l[4] | l[5]) == 0u;
  int shift = 0;
  if (top < (64u << 20)) {  // subnormal entries may be near: scale up, exactly
    shift = 256;
    top = 0u;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const double x = scalbn_rare(a_in[i], shift);
      h[i] = (unsigned)__double2hiint(x);
      l[i] = (unsigned)__double2loint(x);
      top = max(top, h[i] & 0x7fffffffu);
    }
  }
  const int E = (int)(top >> 20);
  F.e = E - 1022 - shift;
  unsigned far = 0u;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const int d = E - (int)((h[i] >> 20) & 0x7ffu);
    const bool zero = i < 3 && ((h[i] << 1) | l[i]) == 0u;
    far = max(far, zero ? 0u : (unsigned)d);
    const int sign = zero ? 0 : (((int)h[i] >> 31) | 1);
    const unsigned m = (h[i] & 0xfffffu) | 0x100000u;  // 53-bit fraction m : l
    const unsigned y1 = __funnelshift_l(l[i], m, 8) >> (d & 31), y0 = __funnelshift_r(l[i] << 8, m << 8 | l[i] >> 24, d);
    F.a[i].h = (int)__funnelshift_r(y0, y1, 31) * sign;
    F.a[i].l = (int)(y0 & 0x7fffffffu) * sign;
  }
  F.similar = far <= kSpread;
  if (kGraded) {
    unsigned m[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) m[i] = h[i] & 0x7fffffffu;
    const unsigned row = min(min(max(max(m[0], m[3]), m[4]), max(max(m[1], m[3]), m[5])), max(max(m[2], m[4]), m[5]));
    const unsigned block = min(min(max(max(m[0], m[1]), m[3]), max(max(m[0], m[2]), m[4])), max(max(m[1], m[2]), m[5]));
    F.similar &= min(row, block) >= top - ((far > kWide ? kGraded6 : kGraded8) << 20);
    F.graded = (int)(row < top - (kGraded6 << 20)) | (int)(block < top - (kGraded6 << 20)) << 1;
  }
  return F;
}

// An eigenvalue below 2^-6 of the largest entry again, from its vector u (whose
// sign is free) and the record: u^T A u / u^T u in integers, A u x 2^113 without
// rounding, the products x 2^116, so to 2^-80 of the largest entry (a vector's
// error enters squared).  Not inlined and in a loop: few matrices need
// it, and it is short so that its instructions arrive quickly (a warp here
// keeps its CTA waiting).
__device__ __noinline__ double small_value(const double* rec, const int e, const double u0, const double u1,
                                           const double u2) {
  const int shift = e + 1022 < 64 ? 256 : 0, E = e + 1022 + shift;  // as fixed_of
  // 53-bit fraction of x, 0 for a zero
  auto fraction = [](const double x) {
    const unsigned h = (unsigned)__double2hiint(x);
    const int64_t m = (int64_t)((uint64_t)((h & 0xfffffu) | 0x100000u) << 32 | (unsigned)__double2loint(x));
    return (h & 0x7ff00000u) == 0u ? 0 : ((int)h < 0 ? -m : m);
  };
  auto exponent = [](const double x) { return (int)((unsigned)__double2hiint(x) >> 20 & 0x7ffu); };
  // u x 2^60 (|u| < 2)
  const int64_t r0 = fraction(u0) << 9 >> min(1024 - exponent(u0), 63),
                r1 = fraction(u1) << 9 >> min(1024 - exponent(u1), 63),
                r2 = fraction(u2) << 9 >> min(1024 - exponent(u2), 63);
  __int128 p = 0, q = 0, n = 0, t = 0;
#pragma unroll 1
  for (int i = 0, j = 0; i < 3;) {
    double x = rec[i == j ? i : i + j + 2];
    if (shift) x = scalbn_rare(x, shift);
    t += ((__int128)fraction(x) * (j == 0 ? r0 : (j == 1 ? r1 : r2))) >> min(E - exponent(x), (int)kSpread + 1);
    if (++j < 3) continue;
    const int64_t r = i == 0 ? r0 : (i == 1 ? r1 : r2);
    p += (__int128)r * (int64_t)(t >> 57);
    q += (__int128)r * ((int64_t)(t >> 25) & 0xffffffffll);
    n += (__int128)r * r;
    t = 0;
    j = 0;
    ++i;
  }
  p += q >> 32;
  // 61 bits of it, x 2^(60 + s), less u^T u - 1
  const int64_t top = (int64_t)(p >> 56), excess = (int64_t)(n >> 60) - (1ll << 60);
  const int s = __clzll((top < 0 ? -top : top) | 1024) - 3;
  const int64_t w = (int64_t)(p >> (56 - s));
  return to_double_int<60>(w - (((w >> 30) * excess) >> 30), e - s);
}

// Eigenvalues l[3] and, with kVectors, eigenvectors U[i*3+k] of a matrix of
// similar entries, without the sign rule; rk[k] is pair k's place in ascending order.
// False when they could not be certified.  rec: its record (kGraded only).
// (The eigenvalues do not depend on kVectors.)
template <bool kVectors, bool kGraded>
__device__ __forceinline__ bool solve(const Fixed& F, const double* rec, double l[3], double U[9], int rk[3]) {
  const Split* const As = F.a;
  float af[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) af[i] = (float)As[i].h * 0x1p-30f;
  const QuatF f = frame32(af);
  const float sc = 0x1p30f * rsqrt32(fmaf(f.w, f.w, fmaf(f.x, f.x, fmaf(f.y, f.y, f.z * f.z))));
  Quat q = {__float2int_rn(f.w * sc), __float2int_rn(f.x * sc), __float2int_rn(f.y * sc), __float2int_rn(f.z * sc)};
  int64_t R[9], N, B[6];
  Split Rs[9];
  // trace of A/2 x 2^61
  const int64_t trace = (((int64_t)As[0].h + As[1].h + As[2].h) << 30) + (((int64_t)As[0].l + As[1].l + As[2].l) >> 1);
  rotation(q, R, N);
#pragma unroll
  for (int i = 0; i < 9; ++i) Rs[i] = split31(R[i]);
  rotated(As, Rs, trace, N, B);
  int p[3];
  if (!small_rotation(B, p)) return false;
  q = normalised(times(q, p));
  rotation(q, R, N);
#pragma unroll
  for (int i = 0; i < 9; ++i) Rs[i] = split31(R[i]);
  rotated(As, Rs, trace, N, B);
  float e01 = to_float(B[1]), e02 = to_float(B[3]), e12 = to_float(B[4]);
  const float off = fmaxf(fabsf(e01), fmaxf(fabsf(e02), fabsf(e12)));
  float w01 = quotient(e01, to_float(B[2] - B[0])), w02 = quotient(e02, to_float(B[5] - B[0])),
        w12 = quotient(e12, to_float(B[5] - B[2]));
  if (!(fabsf(w01) <= kRotMax) && fabsf(e01) <= kNoise) w01 = 0.f;
  if (!(fabsf(w02) <= kRotMax) && fabsf(e02) <= kNoise) w02 = 0.f;
  if (!(fabsf(w12) <= kRotMax) && fabsf(e12) <= kNoise) w12 = 0.f;
  const float big = fmaxf(fabsf(w01), fmaxf(fabsf(w02), fabsf(w12)));
  const float second = fmaxf(fabsf(w01 * e01), fmaxf(fabsf(w02 * e02), fabsf(w12 * e12)));
  const int64_t eta60 = N - (1ll << 60);
  if (eta60 > kNormMax || eta60 < -kNormMax) return false;
  // (the last comparison fails for a NaN among the w, which the maxima drop)
  if (!(off <= kOffMax && big <= kRotMax && second <= kSecond && w01 + w02 + w12 < 1.f)) return false;
  // R is (1 + eta) times a rotation, |eta| < 2^-27: B is divided by (1 + eta)^2
  // and, with the perturbation below, R by 1 + eta.  B is of A/2: at 2^60 its
  // diagonal is the eigenvalues'.
  const int eta58 = (int)((eta60 + 2) >> 2), eta = (eta58 + 1) >> 1;               // x 2^58, x 2^57
  const int shrink = eta58 - (int)((3 * (int64_t)eta * eta + (1ll << 56)) >> 57);  // eta - 3/2 eta^2
  int64_t b[3] = {B[0], B[2], B[5]};
#pragma unroll
  for (int k = 0; k < 3; ++k) b[k] -= ((int64_t)(int)(b[k] >> 31) * shrink) >> 26;
  // The places are those of the values returned: the division truncates, which
  // can change the order of values that agree to 2^-55 of the largest entry.
  const int b10 = b[1] < b[0], b20 = b[2] < b[0], b21 = b[2] < b[1];
  rk[0] = b10 + b20;
  rk[1] = 1 - b10 + b21;
  rk[2] = 2 - b20 - b21;
#pragma unroll
  for (int k = 0; k < 3; ++k) l[k] = to_double_int<60>(b[k], F.e);
  int small = 0;  // bit k: eigenvalue k is to be formed again
  if (kGraded && F.graded) {
#pragma unroll
    for (int k = 0; k < 3; ++k) small |= (int)((uint64_t)(b[k] + kSmall) < (uint64_t)(2 * kSmall)) << k;
    if ((F.graded & 2) && (small & (small - 1))) return false;
    if (!(F.graded & 1)) small = 0;
  }
  if (kVectors || small) {
    // R (I + W + W^2/2 - eta), W antisymmetric: orthogonal to third order.  The
    // factors are held x 2^57 when W is small enough, as it is but for close
    // pairs, else x 2^53.
    const bool fine = big <= 0x1p-27f;
    const float c = fine ? 0x1p57f : 0x1p53f, hc = 0.5f * c;
    const int x01 = __float2int_rn(w01 * c), x02 = __float2int_rn(w02 * c), x12 = __float2int_rn(w12 * c);
    const int scale = fine ? eta : (eta + 8) >> 4;
    const float s02 = w02 * w02, s12 = w12 * w12;
    const int n0 = __float2int_rn(-hc * fmaf(w01, w01, s02)) - scale,
              n1 = __float2int_rn(-hc * fmaf(w01, w01, s12)) - scale,
              n2 = __float2int_rn(-hc * fmaf(w02, w02, s12)) - scale;
    const int y01 = __float2int_rn(-hc * w02 * w12), y02 = __float2int_rn(hc * w01 * w12),
              y12 = __float2int_rn(-hc * w01 * w02);
    const int shift = fine ? 25 : 21;
    const int64_t half = 1ll << (shift - 1);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int r0 = Rs[3 * i].h, r1 = Rs[3 * i + 1].h, r2 = Rs[3 * i + 2].h;  // x 2^29
      const int64_t d0 = madw(r2, y02 - x02, madw(r1, y01 - x01, madw(r0, n0, half)));
      const int64_t d1 = madw(r2, y12 - x12, madw(r1, n1, madw(r0, y01 + x01, half)));
      const int64_t d2 = madw(r2, n2, madw(r1, y12 + x12, madw(r0, y02 + x02, half)));
      U[i * 3 + 0] = to_double_int<61>((R[3 * i] << 1) + (d0 >> shift));
      U[i * 3 + 1] = to_double_int<61>((R[3 * i + 1] << 1) + (d1 >> shift));
      // a third of the conversions on the otherwise idle FP64 pipe (2^22 mixed
      // matrices 522 us, none 530, two thirds 544)
      U[i * 3 + 2] = to_double<61>((R[3 * i + 2] << 1) + (d2 >> shift));
    }
    if (kGraded && small) {
      if (small & 1) l[0] = small_value(rec, F.e, U[0], U[3], U[6]);
      if (small & 2) l[1] = small_value(rec, F.e, U[1], U[4], U[7]);
      if (small & 4) l[2] = small_value(rec, F.e, U[2], U[5], U[8]);
      rk[0] = (int)(l[1] < l[0]) + (int)(l[2] < l[0]);
      rk[1] = (int)(l[0] <= l[1]) + (int)(l[2] < l[1]);
      rk[2] = (int)(l[0] <= l[2]) + (int)(l[1] <= l[2]);
    }
  }
  return true;
}

// Sign rule of column k of U: its largest-magnitude component, the first of
// equals, becomes positive (magnitudes compared as integers, sign bits
// flipped).
__device__ __forceinline__ void sign_rule(double U[9], const int k) {
  const uint64_t m0 = mag_bits(U[k]), m1 = mag_bits(U[3 + k]), m2 = mag_bits(U[6 + k]);
  const double big = (m2 > m0 && m2 > m1) ? U[6 + k] : ((m1 > m0) ? U[3 + k] : U[k]);
  const int flip = __double2hiint(big) & (int)0x80000000;
#pragma unroll
  for (int i = 0; i < 3; ++i) U[i * 3 + k] = flip_sign(U[i * 3 + k], flip);
}

}  // namespace
}  // namespace fx
}  // namespace syev3
