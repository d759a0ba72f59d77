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
  Rot32 J;
  if (q == 0.f) {
    const bool keep = p >= r;
    J.c = keep ? 1.f : 0.f;
    J.s = keep ? 0.f : 1.f;
    J.l1 = keep ? p : r;
    J.l2 = keep ? r : p;
    return J;
  }
  const float D = p - r, q2 = q + q;
  const float rad = sqrt32(fmaf(D, D, q2 * q2));
  const float den = fabsf(D) + rad;
  const float t = (den > 0.f) ? q2 * rcp32(den) : copysignf(1.f, q);
  const bool right = D >= 0.f;
  const float hi = right ? p : r, lo = right ? r : p;
  J.l1 = fmaf(t, q, hi);
  J.l2 = fmaf(-t, q, lo);
  const float k = rsqrt32(fmaf(t, t, 1.f));
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
// (model[k]).  rab = 1/ab.
__device__ __forceinline__ P2 start32x2(const P2 ab, const P2 rab, const P2 b1, const P2 b2, const P2 g, const P2 c,
                                       const P2 K, P2& x7, bool model[2]) {
  const P2 hg = pmul(pp(0.5f), g), bs = padd(b1, b2);
  const P2 rt = psqrt(pfma(hg, hg, bs));
  x7 = psel(g.x >= 0.f, g.y >= 0.f, padd(hg, rt), pmul(bs, prcp(psub(rt, hg))));
  const P2 c2 = pfma(c, rab, pp(1.f));
  const P2 disc = psqrt(pfma(K, K, pmul(pmul(pp(4.f), c2), b1)));
  const bool kx = K.x >= 0.f, ky = K.y >= 0.f;
  const P2 xm = pmul(psel(kx, ky, padd(b1, b1), psub(disc, K)), prcp(psel(kx, ky, padd(K, disc), padd(c2, c2))));
  const P2 r1 = prcp(xm), r2 = prcp(padd(xm, ab));
  const P2 fpm = pfma(pmul(b2, r2), r2, pfma(pmul(b1, r1), r1, pp(1.f)));
  const P2 x0 = padd(xm, pfma(pmul(pmul(padd(c, c), xm), xm), prcp(pmul(pmul(ab, ab), fpm)),
                             pmul(pp(0x1p-20f), xm)));
  model[0] = (xm.x > 0.f) && (xm.x < 0.0625f * ab.x) && (x0.x < x7.x);
  model[1] = (xm.y > 0.f) && (xm.y < 0.0625f * ab.y) && (x0.y < x7.y);
  return psel(model[0], model[1], x0, x7);
}

// The step of bg_step32 for both problems (nb2 = -b2, ng = -g); *fx
// receives f(x).
template <bool kBranchFree>
__device__ __forceinline__ P2 bg_step32x2(const P2 ab, const P2 b1, const P2 b2, const P2 nb2, const P2 ng,
                                         const P2 c, const P2 K, const P2 x, P2* fx) {
  const P2 r1 = prcp(x), r2 = prcp(padd(x, ab));
  const P2 t1 = pmul(b1, r1);
  const bool sx = x.x < ab.x, sy = x.y < ab.y;
  // x + K - b1/x + c x/(x+ab) below ab, x - g - b1/x - b2/(x+ab) above
  const P2 f = padd(psub(padd(x, psel(sx, sy, K, ng)), t1), pmul(psel(sx, sy, pmul(c, x), nb2), r2));
  *fx = f;
  const P2 t2 = pmul(b2, r2);
  const P2 fp = pfma(t2, r2, pfma(t1, r1, pp(1.f)));
  const P2 w0 = pfma(pmul(t2, ab), pmul(r2, r2), pp(1.f));
  const P2 rb = prcp(pfma(f, r1, fp));
  const P2 fr = pmul(f, rb);
  const P2 q = padd(pp(1.f), pmul(pmul(pmul(pp(-4.f), w0), pmul(r1, rb)), fr));
  const P2 delta = pmul(padd(fr, fr), prcp(padd(pp(1.f), psqrt(make_float2(fmaxf(0.f, q.x), fmaxf(0.f, q.y))))));
  P2 xn = psub(x, delta);
  const P2 d2 = padd(delta, delta);  // Delta >= x/2 (exact doubling)
  const bool dx = !(d2.x < x.x), dy = !(d2.y < x.y);
  if constexpr (kBranchFree) {
    // the zero of phi_j for both problems, kept where Delta >= x/2
    const P2 xr = pmul(x, r2);
    const P2 w1 = pfma(pmul(b2, xr), pmul(xr, xr), b1);
    const P2 sg = pfma(w0, x, pmul(pfma(w1, r1, f), pp(-1.f)));
    const P2 rt = psqrt(pfma(sg, sg, pmul(pmul(pp(4.f), w0), w1)));
    const bool px = sg.x > 0.f, py = sg.y > 0.f;
    const P2 xd = pmul(psel(px, py, padd(sg, rt), padd(w1, w1)), prcp(psel(px, py, padd(w0, w0), psub(rt, sg))));
    xn = psel(dx, dy, xd, xn);
  } else {
    if (dx || dy) {  // rare
      if (dx) xn.x = phi_zero32(b1.x, b2.x, x.x, r1.x, r2.x, w0.x, f.x);
      if (dy) xn.y = phi_zero32(b1.y, b2.y, x.y, r1.y, r2.y, w0.y, f.y);
    }
  }
  return psel(f.x > 0.f && xn.x < x.x, f.y > 0.f && xn.y < x.y, xn, x);
}

// mu and nu in FP32 on a fixed schedule, both problems paired: from the
// starts of start32x2 three Borges-Gragg steps, straight-line (no lane
// leaves early, so the warp stays converged; a small-root start found left
// of the root is replaced by the start of Eq. (7) after the first
// evaluation).  The last step moves x by about the error the one before
// left, and the step converges cubically, so a move below kMoveTol x leaves
// an error of order kMoveTol^3 x.  more[k] marks a problem whose last step
// moved x by more than that; the kernel finishes those roots apart from the
// straight-line code (see k_syev3_f32).
__device__ __forceinline__ void roots32x2(const P2 ab, const P2 rab, const P2 b1, const P2 b2, const P2 g,
                                          const P2 c, const P2 K, float x[2], bool more[2]) {
  const P2 nb2 = make_float2(-b2.x, -b2.y), ng = make_float2(-g.x, -g.y);
  P2 x7, f0, f1, f2;
  bool model[2];
  const P2 x0 = start32x2(ab, rab, b1, b2, g, c, K, x7, model);
  P2 x1 = bg_step32x2<true>(ab, b1, b2, nb2, ng, c, K, x0, &f0);
  // the small-root start was not right of the root: restart from Eq. (7)'s
  x1 = psel(model[0] && !(f0.x > 0.f), model[1] && !(f0.y > 0.f), x7, x1);
  const P2 x2 = bg_step32x2<false>(ab, b1, b2, nb2, ng, c, K, x1, &f1);
  const P2 x3 = bg_step32x2<false>(ab, b1, b2, nb2, ng, c, K, x2, &f2);
  const P2 mv = psub(x2, x3), th = pmul(pp(kMoveTol), x3);
  more[0] = mv.x > th.x;
  more[1] = mv.y > th.y;
  x[0] = x3.x;
  x[1] = x3.y;
}

}  // namespace
}  // namespace f32
}  // namespace syev3
