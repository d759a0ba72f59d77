// solve_f32.cuh -- FP32 steps of the method of C. F. Borges (arXiv
// 1806.06698) shared by the FP32 kernels and by the FP32 solve that the FP64
// kernel refines: the ordered Jacobi rotation (Sec. 1) and the Borges-Gragg
// zero finder for mu and nu (Sec. 1.4.1), both problems paired on the packed
// FP32 instructions.
#pragma once

#include <cmath>

#include "arith.cuh"

namespace syev3 {
namespace f32 {
namespace {  // internal linkage: every translation unit gets its own copy

// A last zero-finder move above kMoveTol x (relative error of order
// kMoveTol^3 = 2^-24 after the cubically convergent step) sends the root to
// further steps.
constexpr float kMoveTol = 0x1p-8f;

// Sec. 1: ordered Jacobi rotation of [[p,q],[q,r]] in FP32.
struct Rot32 {
  float c, s, l1, l2;
};

__device__ __forceinline__ Rot32 ordered_rotation32(float p, float q, float r) {
  // (selects, no branch: batches with diagonal matrices would take both sides;
  // 2^23 mixed matrices 179.9 -> 177.4 us together with the paired pre-scale)
  Rot32 J;
  const float D = p - r, q2 = q + q;
  const float rad = sqrt32(fmaf(D, D, q2 * q2));
  const float den = fabsf(D) + rad;
  float t = (den > 0.f) ? q2 * rcp32(den) : copysignf(1.f, q);
  if (q == 0.f) t = 0.f;
  const bool right = D >= 0.f;
  const float hi = right ? p : r, lo = right ? r : p;
  J.l1 = fmaf(t, q, hi);
  J.l2 = fmaf(-t, q, lo);
  float k = rsqrt32(fmaf(t, t, 1.f));
  if (q == 0.f) k = 1.f;
  J.c = right ? k : t * k;
  J.s = right ? t * k : k;
  return J;
}

// The zero of phi_j (the model of Eq. (5) through x) taken directly: the
// root of omega_0 y^2 - sigma y - omega_1 = 0, for a step Delta >= x/2 (a
// start far right of the root).  r1 = 1/x, r2 = 1/(x + ab).
__device__ __forceinline__ float phi_zero32(const float b1, const float b2, const float x, const float r1,
                                            const float r2, const float w0, const float f) {
  const float xr = x * r2;
  const float w1 = fmaf(b2 * xr, xr * xr, b1);
  const float sg = fmaf(w0, x, -fmaf(w1, r1, f));
  const float rt = sqrt32(fmaf(sg, sg, 4.f * w0 * w1));
  return (sg > 0.f) ? (sg + rt) * rcp32(2.f * w0) : (2.f * w1) * rcp32(rt - sg);
}

// Pairs of FP32 values -- .x for the problem of mu, .y for that of nu -- on
// the packed FP32 instructions of sm_100 and later, which perform the same
// correctly rounded operation on both halves: the two problems of a lane run
// the same expressions, so they issue as one instruction stream.  A
// difference a - b is formed as fma(b, -1, a), which rounds the exact
// difference once, as a subtraction does.  Reciprocals, roots, comparisons
// and selections stay per half.
using P2 = float2;
__device__ __forceinline__ P2 pp(const float a) { return make_float2(a, a); }
__device__ __forceinline__ P2 padd(const P2 a, const P2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ P2 psub(const P2 a, const P2 b) { return __ffma2_rn(b, pp(-1.f), a); }
__device__ __forceinline__ P2 pmul(const P2 a, const P2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ P2 pfma(const P2 a, const P2 b, const P2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ P2 prcp(const P2 a) { return make_float2(rcp32(a.x), rcp32(a.y)); }
__device__ __forceinline__ P2 psqrt(const P2 a) { return make_float2(sqrt32(a.x), sqrt32(a.y)); }
__device__ __forceinline__ P2 psel(const bool px, const bool py, const P2 a, const P2 b) {
  return make_float2(px ? a.x : b.x, py ? a.y : b.y);
}

// The starts of f64::start32 (solve_f64.cuh) for both problems: the zero x7 of the limit
// model of Eq. (7), and the small-root model's start taken where it applies
// (model[k]; xm < ab/16).  Its second-order term 2 c xm^2 / (ab^2 f'(xm)) is
// taken with f' = 1, its lower bound: x0 only moves further right, which
// saves three reciprocals, and the share of matrices with a root left to
// further steps stays (gaussian entries 0.26 %, mixed 0.19 -> 0.20 %).
// rab = 1/ab.
__device__ __forceinline__ P2 start32x2(const P2 ab, const P2 rab, const P2 b1, const P2 b2, const P2 g, const P2 c,
                                       const P2 K, P2& x7, bool model[2]) {
  const P2 hg = pmul(pp(0.5f), g), bs = padd(b1, b2);
  const P2 rt = psqrt(pfma(hg, hg, bs));
  x7 = psel(g.x >= 0.f, g.y >= 0.f, padd(hg, rt), pmul(bs, prcp(psub(rt, hg))));
  const P2 c2 = pfma(c, rab, pp(1.f));
  const P2 disc = psqrt(pfma(K, K, pmul(pmul(pp(4.f), c2), b1)));
  const bool kx = K.x >= 0.f, ky = K.y >= 0.f;
  const P2 xm = pmul(psel(kx, ky, padd(b1, b1), psub(disc, K)), prcp(psel(kx, ky, padd(K, disc), padd(c2, c2))));
  const P2 y = pmul(xm, rab);
  const P2 x0 = pfma(padd(c, c), pmul(y, y), pfma(xm, pp(0x1p-20f), xm));
  model[0] = (xm.x > 0.f) && (xm.x < 0.0625f * ab.x) && (x0.x < x7.x);
  model[1] = (xm.y > 0.f) && (xm.y < 0.0625f * ab.y) && (x0.y < x7.y);
  return psel(model[0], model[1], x0, x7);
}

// f and the parts of the model phi_j at x for both problems (nb2 = -b2,
// ng = -g): f = x + K - b1/x + c x/(x+ab) below ab, x - g - b1/x - b2/(x+ab)
// above; r1 = 1/x, r2 = 1/(x+ab), t1 = b1 r1, t2 = b2 r2.
struct At32 {
  P2 r1, r2, t1, t2, w0, f;
};
__device__ __forceinline__ At32 at32x2(const P2 ab, const P2 b1, const P2 b2, const P2 nb2, const P2 ng,
                                      const P2 c, const P2 K, const P2 x) {
  At32 m;
  m.r1 = prcp(x);
  m.r2 = prcp(padd(x, ab));
  m.t1 = pmul(b1, m.r1);
  m.t2 = pmul(b2, m.r2);
  const bool sx = x.x < ab.x, sy = x.y < ab.y;
  m.f = padd(psub(padd(x, psel(sx, sy, K, ng)), m.t1), pmul(psel(sx, sy, pmul(c, x), nb2), m.r2));
  m.w0 = pfma(pmul(m.t2, ab), pmul(m.r2, m.r2), pp(1.f));
  return m;
}

// A Borges-Gragg step with the zero of phi_j taken directly (phi_zero32) for
// both problems; x itself where f(x) <= 0.
__device__ __forceinline__ P2 direct_step32x2(const P2 b1, const P2 b2, const P2 x, const At32& m) {
  const P2 xr = pmul(x, m.r2);
  const P2 w1 = pfma(pmul(b2, xr), pmul(xr, xr), b1);
  const P2 sg = pfma(m.w0, x, pmul(pfma(w1, m.r1, m.f), pp(-1.f)));
  const P2 rt = psqrt(pfma(sg, sg, pmul(pmul(pp(4.f), m.w0), w1)));
  const bool px = sg.x > 0.f, py = sg.y > 0.f;
  const P2 xd = pmul(psel(px, py, padd(sg, rt), padd(w1, w1)), prcp(psel(px, py, padd(m.w0, m.w0), psub(rt, sg))));
  return psel(m.f.x > 0.f && xd.x < x.x, m.f.y > 0.f && xd.y < x.y, xd, x);
}

// mu and nu in FP32 on a fixed schedule, both problems paired and
// straight-line (no lane leaves early, so the warp stays converged): from the
// starts of start32x2 two steps that take the model's zero directly -- valid
// from any distance; its rounding errors, a few units of the root, are left
// to the last step -- and one in the form of Eq. (6), x - Delta.  A small-root
// start found left of the root is replaced by the start of Eq. (7) after the
// first evaluation.  In the last step 2/(1 + sqrt(1 + z)), z = -4 w0 f/(x D^2)
// with D = f/x + f', is its series 1 - z/4 + z^2/8: kept where |Delta| is at
// most kMoveTol x, so |z| <= 2^-6 (f' >= w0) and the rest, below 5/64 |z|^3,
// moves the root by less than 2^-29 of itself; the step's own error there is
// of order kMoveTol^3 (0.25 x 2^-24 at most over 4e6 sampled spikes and gaps,
// with the root or with the series).  A root that the second step left on the
// left by its rounding is corrected from there.  more[k] marks a problem whose
// last step is longer than that; the kernel finishes those roots apart from
// the straight-line code (see k_syev3_f32).
//
// Instruction issue and the MUFU unit bound these steps: 5 reciprocals and
// roots per step and problem in the form of Eq. (6), and 7 where both forms
// are computed, against 4 in each of the first two steps and 3 in the last.
// FP32 solve of 2^23 mixed matrices 205.1 -> 186.2 us, eigenvalues only
// 164.7 -> 145.6 us, the FP64 solve's start 2 % of that kernel.
__device__ __forceinline__ void roots32x2(const P2 ab, const P2 rab, const P2 b1, const P2 b2, const P2 g,
                                          const P2 c, const P2 K, float x[2], bool more[2]) {
  const P2 nb2 = make_float2(-b2.x, -b2.y), ng = make_float2(-g.x, -g.y);
  P2 x7;
  bool model[2];
  const P2 x0 = start32x2(ab, rab, b1, b2, g, c, K, x7, model);
  const At32 m0 = at32x2(ab, b1, b2, nb2, ng, c, K, x0);
  P2 x1 = direct_step32x2(b1, b2, x0, m0);
  // the small-root start was not right of the root: restart from Eq. (7)'s
  x1 = psel(model[0] && !(m0.f.x > 0.f), model[1] && !(m0.f.y > 0.f), x7, x1);
  const P2 x2 = direct_step32x2(b1, b2, x1, at32x2(ab, b1, b2, nb2, ng, c, K, x1));
  const At32 m = at32x2(ab, b1, b2, nb2, ng, c, K, x2);
  const P2 rb = prcp(pfma(m.f, m.r1, pfma(m.t2, m.r2, pfma(m.t1, m.r1, pp(1.f)))));
  const P2 fr = pmul(m.f, rb), z = pmul(pmul(pmul(pp(-4.f), m.w0), pmul(m.r1, rb)), fr);
  const P2 delta = pfma(pmul(fr, z), pfma(z, pp(0.125f), pp(-0.25f)), fr);
  const P2 x3 = psub(x2, delta), th = pmul(pp(kMoveTol), x2);
  const bool near_x = fabsf(delta.x) <= th.x, near_y = fabsf(delta.y) <= th.y;
  const bool right_x = m.f.x > 0.f, right_y = m.f.y > 0.f;
  more[0] = right_x && !near_x;
  more[1] = right_y && !near_y;
  x[0] = (near_x || (right_x && x3.x < x2.x)) ? x3.x : x2.x;
  x[1] = (near_y || (right_y && x3.y < x2.y)) ? x3.y : x2.y;
}

}  // namespace
}  // namespace f32
}  // namespace syev3
