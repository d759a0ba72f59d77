// syev3_f32.cu -- FP32 batched 3x3 symmetric eigensolver for sm_103a, plain
// and compensated (the precision form).
//
// The steps are those of the FP64 solver (C. F. Borges, arXiv 1806.06698,
// Secs. 1-1.4.1) carried out in FP32: ordered Jacobi rotation to an arrow,
// the deflation test, the deflated 2x2 solve or the Borges-Gragg zero finder
// for mu and nu, the trace identity and the closed-form eigenvectors.  The
// spectral function is evaluated in the cancellation-free form for x < abar
// (see solve_f64.cuh).
//
// The compensated form (SYEV3_F32_COMPENSATED) adds, in FP32:
//  * the deflation test of Sec. 1.1 decided as on exact products, so the
//    decision is not blurred by FP32 rounding: on the FP32 sides where they
//    are clearly apart, with double-float (error-free transformation)
//    products where they are close;
//  * a double-float evaluation of the spectral function at the FP32 root
//    and one Newton correction (Sec. 1.4.2) with it,
// and refines the matrices it flags -- near-deflated (the test's two sides
// within a factor kNearDefl), clustered (a relative eigenvalue gap below
// kClusterTau) or capped -- from their input records: in 62-bit fixed point
// (solve_fx.cuh), or, for graded or structured ones, by a final FP64 Newton
// step on mu and nu and eigenvectors re-formed (and so re-orthogonalised) in
// FP64; an FP64 residual check against the input feeds the counters.  A CTA
// lists its flagged matrices in shared memory and refines them in whole warps
// after its last tile; no global scratch memory is used (syev3_batched_ws
// lists them in its workspace instead and refines them with a second kernel
// for large batches).
//
// The two root problems of a lane (mu and nu) run the same expressions, so
// their arithmetic is paired on the packed FP32 instructions (two correctly
// rounded operations per instruction); reciprocals, roots, comparisons and
// selections stay per half.  Lanes of the three classes (diagonal, deflated,
// reduced) in one warp take different branches of the solve; an explicit
// __syncwarp over the lanes that form eigenpairs rejoins them for the common
// tail (without it the warp was measured to stay split there).
//
// Memory path: tiles of kTPB records (24 B each) by 1-D bulk copy into shared
// memory, double-buffered on mbarriers; a full tile's results leave their
// staging rows by bulk copy too, so that no thread loads and stores them and
// one barrier per tile fewer is needed (2^24 mixed matrices, plain: 415 us
// against 484 with 16-byte stores by all threads).  The plain form moves 72 B
// per matrix; it is bound by instruction issue (17.7 warp instructions per
// matrix, 72 % of the slots), not by HBM.

#include <cmath>
#include <cstdint>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "serve_tile.cuh"
#include "solve_f32.cuh"
#include "solve_f64.cuh"
#include "solve_fx.cuh"

namespace syev3 {
namespace {

using namespace f32;

constexpr int kTPB = 128;
constexpr int kMaxIt32 = 32;              // FP32 zero-finder step cap
constexpr float kEps32 = 0x1p-23f;
constexpr float kCDefl32 = 1.0f;          // C of the deflation test (Sec. 1.1)
constexpr float kCTerm32 = 2.0f;          // C of the stopping rule (Sec. 1.4.1)
constexpr float kTinySpike32 = 0x1p-60f;  // spikes below this are zeroed (beta-deflation)
// The lanes refined are those FP32 cannot resolve: a deflation test
// whose two sides lie within a factor kNearDefl of each other (the decision
// rests on the last bits of the FP32 data), or a relative eigenvalue gap
// below kClusterTau = one unit of FP32 resolution (the pair's eigenvectors are
// then not determined by FP32 arithmetic).  A sweep of both on the mixed and
// structure-tensor batches found every subset's error against the FP64
// oracle within 2.1 eps32 ||A||_F (eigenvalues), 2.9 (residual) and 7.6
// (orthogonality) for every setting, far inside the 64 eps32 bar; wider
// windows only cost time (a factor 16 window flagged 16 % of the mixed batch).
constexpr float kNearDefl = 2.0f;         // near-deflated: test sides within this factor
constexpr float kClusterTau = 0x1p-23f;   // clustered: relative gap below this
constexpr double kResidualTol = 16.0 * 0x1p-23;  // FP64 residual check, times ||A||_F
constexpr int kPlain = 0, kComp32 = 1, kDeferred = 2;  // modes of k_syev3_f32

constexpr int kDiag = f64::kDiagonal, kDefl = f64::kDeflated, kRed = f64::kReduced,
              kNonFin = f64::kNonFinite, kIdle = f64::kIdle;

__device__ unsigned g_flags32;

struct Lane32 {
  float a1, a2, b1, b2, g, c, s;  // ordered arrow and rotation (pre-scaled frame)
  int e;                          // A was divided by 2^e
  int cls;
  bool near_defl;
};

template <bool kComp>
__device__ __forceinline__ Lane32 make_lane32(const float a_in[6]) {
  Lane32 L;
  L.near_defl = false;
  // largest |a_ij| as a bit pattern, NaN above all (3 instructions; by integer
  // maxima 11, 1.3 % of the kernel together with the ranks of finish32)
  const unsigned mag = __float_as_uint(
      max_abs3(max_abs3(a_in[0], a_in[1], a_in[2]), max_abs3(a_in[3], a_in[4], a_in[5]), 0.f));
  if (mag >= 0x7f800000u) {  // an infinite or NaN entry
    L.cls = kNonFin;
    return L;
  }
  const int E = (int)(mag >> 23);
  float a[6];
  if (E >= 1 && E <= 252) {  // exact power-of-two pre-scale: largest entry in [0.5, 1)
    L.e = E - 126;
    const float sc = pow2f(-L.e);
#pragma unroll
    for (int i = 0; i < 6; i += 2) {
      const P2 y = pmul(make_float2(a_in[i], a_in[i + 1]), pp(sc));
      a[i] = y.x;
      a[i + 1] = y.y;
    }
  } else {
    float amax = 0.f;
#pragma unroll
    for (int i = 0; i < 6; ++i) amax = fmaxf(amax, fabsf(a_in[i]));
    int e = 0;
    if (amax > 0.f) frexpf(amax, &e);
    L.e = e;
#pragma unroll
    for (int i = 0; i < 6; ++i) a[i] = scalbnf(a_in[i], -e);
  }
  const Rot32 J = ordered_rotation32(a[0], a[3], a[1]);
  L.a1 = J.l1;
  L.a2 = J.l2;
  L.c = J.c;
  L.s = J.s;
  L.g = a[2];
  float b1 = fmaf(J.c, a[4], J.s * a[5]);
  float b2 = fmaf(J.c, a[5], -J.s * a[4]);
  if (fabsf(b1) < kTinySpike32) b1 = 0.f;
  if (fabsf(b2) < kTinySpike32) b2 = 0.f;
  L.b1 = b1;
  L.b2 = b2;
  if (b1 == 0.f && b2 == 0.f) {
    L.cls = kDiag;
    return L;
  }
  // Sec. 1.1: |abar b1 b2| <= C eps |a1 + a2| h^2.
  const float h2 = fmaf(b1, b1, b2 * b2);
  const float lhs = fabsf((L.a1 - L.a2) * b1 * b2);
  const float rhs = (kCDefl32 * kEps32) * fabsf(L.a1 + L.a2) * h2;
  if (kComp) {
    // The decision of the exact sides (exact arithmetic on the FP32 arrow).
    // The FP32 sides above carry 3 and 4 roundings, a relative error below
    // 7 x 2^-24 together, and every intermediate is normal when both sides
    // are >= 2^-120; sides further apart than a factor 1 + 2^-20 (one more
    // rounding in forming the bounds) are therefore ordered as the exact
    // ones.  Closer sides, or sides near underflow, are decided with
    // double-float products, which carry the exact sides to ~2^-46.
    const bool clear = lhs >= 0x1p-120f && rhs >= 0x1p-120f &&
                       (lhs <= rhs * (1.f - 0x1p-20f) || lhs >= rhs * (1.f + 0x1p-20f));
    if (clear) {
      L.cls = (lhs <= rhs) ? kDefl : kRed;
    } else {
      const F2 ab = two_sum(L.a1, -L.a2);
      const F2 dl = ff_mul1(ff_mul1(ab, b1), b2);
      const F2 sum12 = two_sum(L.a1, L.a2);
      const F2 dh2 = ff_add(two_prod(b1, b1), two_prod(b2, b2));
      F2 dr = ff_mul(sum12, dh2);
      dr.h *= kCDefl32 * kEps32;
      dr.l *= kCDefl32 * kEps32;
      const F2 al = {fabsf(dl.h), dl.h < 0.f ? -dl.l : dl.l};
      const F2 ar = {fabsf(dr.h), dr.h < 0.f ? -dr.l : dr.l};
      L.cls = ff_le(al, ar) ? kDefl : kRed;
    }
    L.near_defl = (lhs < kNearDefl * rhs) && (lhs * kNearDefl > rhs);
  } else {
    L.cls = (lhs <= rhs) ? kDefl : kRed;
  }
  return L;
}

// One Borges-Gragg step in FP32 (Sec. 1.4.1) from x: returns x_{j+1}, or x
// itself when f(x) <= 0 (at or past the root: rounding level).  For x < ab,
// f = x + K - b1/x + c x/(x+ab) (the cancellation-free form); x_{j+1} is
// x - Delta (Eq. (6)), or the zero of phi_j taken directly when Delta >= x/2.
// *fx receives f(x).
__device__ __forceinline__ float bg_step32(const float ab, const float b1, const float b2, const float g,
                                          const float c, const float K, const float x, float* fx,
                                          float* fpx = nullptr) {
  const float r1 = rcp32(x), r2 = rcp32(x + ab);
  const float t1 = b1 * r1, t2 = b2 * r2;
  const bool small = x < ab;
  const float f = ((x + (small ? K : -g)) - t1) + (small ? c * x * r2 : -t2);
  *fx = f;
  const float fp = fmaf(t2, r2, fmaf(t1, r1, 1.f));
  if (fpx) *fpx = fp;
  const float w0 = fmaf(t2 * ab, r2 * r2, 1.f);
  const float rb = rcp32(fmaf(f, r1, fp));
  const float fr = f * rb;
  const float z = (-4.f * w0) * (r1 * rb) * fr;
  const float delta = 2.f * fr * rcp32(1.f + sqrt32(fmaxf(0.f, 1.f + z)));
  float xn = x - delta;
  if (!(delta < 0.5f * x)) xn = phi_zero32(b1, b2, x, r1, r2, w0, f);  // rare
  return (f > 0.f && xn < x) ? xn : x;
}

// Further steps for one problem until f/f' < C eps32 x (Sec. 1.4.1), f <= 0
// or a stalled step; returns false if kMaxIt32 steps were not enough.  Not
// inlined: it runs for few roots, and inlined it would weigh on the
// registers and scheduling of the kernel's main path.
__device__ __noinline__ bool roots32_more(const float ab, const float b1, const float b2, const float g, float* x) {
  const float c = b2 * rcp32(ab), K = -g - c;
  for (int it = 0; it < kMaxIt32; ++it) {
    float f, fp;
    const float xn = bg_step32(ab, b1, b2, g, c, K, *x, &f, &fp);
    const bool go = f > (kCTerm32 * kEps32) * (*x) * fp && xn < *x;  // f/f' >= C eps x: not yet
    *x = xn;
    if (!go) return true;
  }
  return false;
}

// The two problems' data of a reduced arrow (Sec. 1.2): problem 0 (mu)
// has spikes (b1^2, b2^2) and gap g - a1, problem 1 (nu) the spikes swapped
// and a2 - g; ab = a1 - a2.
__device__ __forceinline__ void roots_setup32(const Lane32& L, const float ab, float b1[2], float b2[2],
                                              float g[2]) {
  (void)ab;
  const P2 bb = pmul(make_float2(L.b1, L.b2), make_float2(L.b1, L.b2));
  const P2 gg = psub(make_float2(L.g, L.a2), make_float2(L.a1, L.g));
  b1[0] = bb.x; b1[1] = bb.y; b2[0] = bb.y; b2[1] = bb.x;
  g[0] = gg.x; g[1] = gg.y;
}

// Double-float value of the spectral function at both roots x (FP32 data
// exact), and one Newton correction x - f/f' with it (Sec. 1.4.2).  Each
// term is formed as an unevaluated pair (head, low part) without
// renormalisation, and the terms are added by cascaded summation (Ogita, Rump
// and Oishi 2005, "Sum2"): the heads with TwoSum, every rounding error and
// low part in one FP32 sum, so f comes out as if summed in twice the working
// precision and rounded once.  Data pairs (ab, b1, b2, -g, c, K) need not be
// normalised.
__device__ __forceinline__ P2 pneg(const P2 a) { return pmul(a, pp(-1.f)); }

__device__ __forceinline__ void ptwo_sum(const P2 a, const P2 b, P2& s, P2& e) {
  s = padd(a, b);
  const P2 bb = psub(s, a);
  e = padd(psub(a, psub(s, bb)), psub(b, bb));
}

__device__ __forceinline__ P2 newton_ff2(const P2 abh, const P2 abl, const P2 b1h, const P2 b1l, const P2 b2h,
                                        const P2 b2l, const P2 ngh, const P2 ngl, const P2 ch, const P2 cl,
                                        const P2 Kh, const P2 Kl, const P2 x) {
  const P2 r1 = prcp(x), nx = pneg(x);
  P2 sh, s0l;
  ptwo_sum(x, abh, sh, s0l);
  const P2 sl = padd(s0l, abl);  // x + ab = sh + sl
  const P2 r2 = prcp(sh);
  // b1 / x: the quotient's head and the remainder over x.
  const P2 q1 = pmul(b1h, r1);
  const P2 q1l = pmul(padd(pfma(q1, nx, b1h), b1l), r1);
  // Last term: + c x / (x + ab) below ab (the cancellation-free form),
  // - b2 / (x + ab) above; numerator (nh, nl), quotient (q2, q2l).
  const bool sx = x.x < abh.x, sy = x.y < abh.y;
  const P2 cx = pmul(ch, x);
  const P2 nh = psel(sx, sy, cx, b2h);
  const P2 nl = psel(sx, sy, pfma(cl, x, pfma(ch, x, pneg(cx))), b2l);
  const P2 q2 = pmul(nh, r2), nq2 = pneg(q2);
  const P2 q2l = pmul(pfma(nq2, sl, padd(pfma(nq2, sh, nh), nl)), r2);
  const P2 sg = psel(sx, sy, pp(1.f), pp(-1.f));
  const P2 th = pmul(q2, sg), tl = pmul(q2l, sg);
  const P2 lh = psel(sx, sy, Kh, ngh), ll = psel(sx, sy, Kl, ngl);
  // Sum2 over x + lead - b1/x + last.
  P2 uh, ul, vh, vl, wh, wl;
  ptwo_sum(x, lh, uh, ul);
  vh = psub(uh, q1);  // TwoSum(u.h, -q1)
  {
    const P2 bb = psub(vh, uh);
    vl = psub(psub(uh, psub(vh, bb)), padd(q1, bb));
  }
  ptwo_sum(vh, th, wh, wl);
  const P2 f = padd(wh, padd(padd(padd(ul, vl), padd(wl, ll)), psub(tl, q1l)));
  const P2 fp = pfma(pmul(b2h, r2), r2, pfma(q1, r1, pp(1.f)));
  const P2 xn = pfma(pneg(f), prcp(fp), x);
  return psel(xn.x > 0.f, xn.y > 0.f, xn, x);
}

// The roots (Sec. 1.2) of a lane: root[0] = mu, root[1] = nu (0 for the other
// classes); with kComp, after one Newton correction in double-float.  Returns
// whether the zero finder hit its step cap.  Every lane of the warp calls it.
template <bool kComp>
__device__ __forceinline__ bool roots_of(const Lane32& L, float root[2]) {
  root[0] = root[1] = 0.f;
  bool capped = false;
  bool more[2] = {false, false};
  float ab = 0.f, pb1[2] = {0.f, 0.f}, pb2[2] = {0.f, 0.f}, pg[2] = {0.f, 0.f};
  if (L.cls == kRed) {
    ab = L.a1 - L.a2;
    roots_setup32(L, ab, pb1, pb2, pg);
    const P2 rab = pp(rcp32(ab)), b1p = make_float2(pb1[0], pb1[1]), b2p = make_float2(pb2[0], pb2[1]);
    const P2 g2 = make_float2(pg[0], pg[1]);
    const P2 pc = pmul(b2p, rab);
    roots32x2(pp(ab), rab, b1p, b2p, g2, pc, psub(make_float2(-g2.x, -g2.y), pc), root, more);
  }
  // Rare: roots still moving after the straight-line steps, finished in
  // their own lanes (the warp runs this only when one of its roots needs it).
  if (__any_sync(0xffffffffu, more[0] || more[1])) {
    float xa = root[0], xb = root[1];
    bool ca = false, cb = false;
    if (more[0]) ca = !roots32_more(ab, pb1[0], pb2[0], pg[0], &xa);
    if (more[1]) cb = !roots32_more(ab, pb1[1], pb2[1], pg[1], &xb);
    root[0] = xa;
    root[1] = xb;
    capped = ca || cb;
  }
  if (kComp && L.cls == kRed) {
    // Exact FP32 data as double-float, then one Newton correction with a
    // double-float f at each root (both problems paired).
    const F2 abf = two_sum(L.a1, -L.a2);
    const P2 abh = pp(abf.h), abl = pp(abf.l), rabh = pp(rcp32(abf.h));
    // spikes (b1^2, b2^2) exactly; problem 1 has them swapped
    const P2 Bs = make_float2(L.b1, L.b2);
    const P2 bh = pmul(Bs, Bs), bl = pfma(Bs, Bs, pneg(bh));
    const P2 sbh = make_float2(bh.y, bh.x), sbl = make_float2(bl.y, bl.x);
    P2 gh, gl;  // (g - a1, a2 - g) exactly
    ptwo_sum(make_float2(L.g, L.a2), make_float2(-L.a1, -L.g), gh, gl);
    // c = b2 / abar and K = -(g + c) as unnormalised pairs.
    const P2 ch = pmul(sbh, rabh);
    const P2 cl = pmul(pfma(pneg(ch), abl, padd(pfma(pneg(ch), abh, sbh), sbl)), rabh);
    P2 th, tl;
    ptwo_sum(gh, ch, th, tl);
    const P2 Kh = pneg(th), Kl = pneg(padd(padd(tl, gl), cl));
    const P2 xr = newton_ff2(abh, abl, bh, bl, sbh, sbl, pneg(gh), pneg(gl), ch, cl, Kh, Kl,
                             make_float2(root[0], root[1]));
    root[0] = xr.x;
    root[1] = xr.y;
  }
  return capped;
}

// The sign bit of the largest-magnitude component, the first of equals.
__device__ __forceinline__ unsigned sign_of_largest(const float y0, const float y1, const float y2) {
  float big = (fabsf(y1) > fabsf(y0)) ? y1 : y0;
  big = (fabsf(y2) > fabsf(big)) ? y2 : big;
  return __float_as_uint(big) & 0x80000000u;
}

// Eigenvalues only: those of finish32 (the same expressions, compare order
// and tie rule), ascending, in the scaled frame.
__device__ __forceinline__ void finish32_values(const Lane32& L, float mu, float nu, float l_out[3],
                                                const unsigned sync_mask) {
  const float a1 = L.a1, a2 = L.a2, b1 = L.b1, b2 = L.b2, g = L.g;
  float l0, l1, l2;
  if (L.cls == kDiag) {
    l0 = a1; l1 = a2; l2 = g;
  } else if (L.cls == kDefl) {
    const float h2 = fmaf(b1, b1, b2 * b2);
    const float rh = rsqrt32(h2), h = h2 * rh;
    const float gs = b1 * rh, gc = b2 * rh;
    l0 = fmaf(a1 * gc, gc, a2 * gs * gs);
    const Rot32 K = ordered_rotation32(fmaf(a1 * gs, gs, a2 * gc * gc), h, g);
    l1 = K.l1; l2 = K.l2;
  } else {
    l0 = a1 + mu;
    l1 = (nu - mu) + g;
    l2 = a2 - nu;
  }
  __syncwarp(sync_mask);  // the classes' lanes rejoin
  float t;
  if (l1 < l0) { t = l0; l0 = l1; l1 = t; }
  if (l2 < l1) { t = l1; l1 = l2; l2 = t; }
  if (l1 < l0) { t = l0; l0 = l1; l1 = t; }
  l_out[0] = l0; l_out[1] = l1; l_out[2] = l2;
}

// Eigenpairs of a classified lane in FP32 (scaled frame): eigenvalues in
// l_out[], vectors as columns in U[i*3+k], their ascending ranks in rk[].  The
// kernel is bound by instruction issue, so the vectors 0 and 2 are formed in
// pairs (2^23 mixed matrices 183.5 -> 179.9 us).
__device__ __forceinline__ void finish32(const Lane32& L, float mu, float nu, float l_out[3], float U[9], int rk[3],
                                         const unsigned sync_mask) {
  const float a1 = L.a1, a2 = L.a2, b1 = L.b1, b2 = L.b2, g = L.g;
  float l[3], v1[3];
  P2 w[3];  // components of the vectors 0 (.x) and 2 (.y)
  if (L.cls == kDiag) {
    l[0] = a1; l[1] = a2; l[2] = g;
    w[0] = make_float2(1.f, 0.f); w[1] = make_float2(0.f, 0.f); w[2] = make_float2(0.f, 1.f);
    v1[0] = 0.f; v1[1] = 1.f; v1[2] = 0.f;
  } else if (L.cls == kDefl) {
    const float h2 = fmaf(b1, b1, b2 * b2);
    const float rh = rsqrt32(h2), h = h2 * rh;
    const float gs = b1 * rh, gc = b2 * rh;
    l[0] = fmaf(a1 * gc, gc, a2 * gs * gs);
    const float d2 = fmaf(a1 * gs, gs, a2 * gc * gc);
    const Rot32 K = ordered_rotation32(d2, h, g);
    l[1] = K.l1; l[2] = K.l2;
    v1[0] = gs * K.c; v1[1] = gc * K.c; v1[2] = K.s;
    w[0] = make_float2(gc, -gs * K.s); w[1] = make_float2(-gs, -gc * K.s); w[2] = make_float2(0.f, K.c);
  } else {
    l[0] = a1 + mu;
    l[1] = (nu - mu) + g;
    l[2] = a2 - nu;
    const P2 r = make_float2(mu, nu), pa = padd(r, pp(a1 - a2));
    w[0] = pmul(pp(b1), make_float2(pa.x, r.y));
    w[1] = pmul(pp(b2), make_float2(r.x, pa.y));
    w[2] = pmul(make_float2(r.x, -r.y), pa);
    v1[0] = v1[1] = v1[2] = 0.f;  // u2 = u1 x u3, formed below in the input frame
    P2 ss = pfma(w[0], w[0], pfma(w[1], w[1], pmul(w[2], w[2])));
    if (!(fminf(ss.x, ss.y) >= 0x1p-100f)) {  // squares near underflow: exact power-of-two rescale
      P2 sc = pp(1.f);
      int E0 = 1, E2 = 1;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        E0 = max(E0, (__float_as_int(w[i].x) >> 23) & 0xff);
        E2 = max(E2, (__float_as_int(w[i].y) >> 23) & 0xff);
      }
      if (!(ss.x >= 0x1p-100f)) sc.x = pow2f(126 - E0);
      if (!(ss.y >= 0x1p-100f)) sc.y = pow2f(126 - E2);
#pragma unroll
      for (int i = 0; i < 3; ++i) w[i] = pmul(w[i], sc);
      ss = pfma(w[0], w[0], pfma(w[1], w[1], pmul(w[2], w[2])));
    }
    const P2 inv = make_float2(rsqrt32(ss.x), rsqrt32(ss.y));
#pragma unroll
    for (int i = 0; i < 3; ++i) w[i] = pmul(w[i], inv);
  }
  __syncwarp(sync_mask);  // the three classes' lanes rejoin for the common tail
  float x[3][3];
  {
    const P2 c2 = pp(L.c), y0 = pfma(c2, w[0], pmul(pp(-L.s), w[1])), y1 = pfma(pp(L.s), w[0], pmul(c2, w[1]));
    x[0][0] = y0.x; x[0][1] = y1.x; x[0][2] = w[2].x;
    x[2][0] = y0.y; x[2][1] = y1.y; x[2][2] = w[2].y;
  }
  if (L.cls == kRed) {
    // u2 is the cross product of u1 and u3 (Sec. 1.3), of the normalised
    // vectors and in the input frame ((J u1) x (J u3) = J (u1 x u3)): no
    // normalisation and no back-transform of its own.
    x[1][0] = fmaf(x[0][1], x[2][2], -x[0][2] * x[2][1]);
    x[1][1] = fmaf(x[0][2], x[2][0], -x[0][0] * x[2][2]);
    x[1][2] = fmaf(x[0][0], x[2][1], -x[0][1] * x[2][0]);
  } else {
    x[1][0] = fmaf(L.c, v1[0], -L.s * v1[1]);
    x[1][1] = fmaf(L.s, v1[0], L.c * v1[1]);
    x[1][2] = v1[2];
  }
  // Stable ascending ranks of the three eigenvalues (strict "<" for the
  // later index keeps equal values in branch order); the caller stores each
  // eigenpair at its rank.
  const int p = l[1] < l[0], q = l[2] < l[0], r = l[2] < l[1];
  rk[0] = p + q;
  rk[1] = 1 - p + r;
  rk[2] = 2 - q - r;
  // Sign rule: each vector's largest-magnitude component (the first of
  // equals) made positive, by XOR-ing its sign bits with that component's
  // (never zero: at least 1/sqrt(3) in a unit vector).
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float y0 = x[k][0], y1 = x[k][1], y2 = x[k][2];
    const unsigned sb = sign_of_largest(y0, y1, y2);
    l_out[k] = l[k];
    U[0 * 3 + k] = __uint_as_float(__float_as_uint(y0) ^ sb);
    U[1 * 3 + k] = __uint_as_float(__float_as_uint(y1) ^ sb);
    U[2 * 3 + k] = __uint_as_float(__float_as_uint(y2) ^ sb);
  }
}

// Eigenvalues back to the input's scale, l * 2^e: one exact multiply when
// 2^e is a normal float, scalbnf otherwise (the range check once per lane).
__device__ __forceinline__ void unscale3(float l[3], int e) {
  if (e >= -126 && e <= 127) {
    const float sc = pow2f(e);
#pragma unroll
    for (int k = 0; k < 3; ++k) l[k] *= sc;
  } else {
#pragma unroll
    for (int k = 0; k < 3; ++k) l[k] = scalbnf(l[k], e);
  }
}

// The FP64 residual check ||A u - lambda u|| <= 16 eps32 ||A||_F of a refined
// lane against its input record; true when it fails, for a vector that is not
// of unit length (a zero vector has no residual) and for a NaN.
__device__ __forceinline__ bool residual_fails(const float rec[6], const double lam[3], const double U[9]) {
  const double M[3][3] = {{rec[0], rec[3], rec[4]}, {rec[3], rec[1], rec[5]}, {rec[4], rec[5], rec[2]}};
  double nA = 0.0;
  bool ok = true;
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int q = 0; q < 3; ++q) nA = fma(M[r][q], M[r][q], nA);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double rr = 0.0;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const double v = fma(M[r][0], U[k], fma(M[r][1], U[3 + k], fma(M[r][2], U[6 + k], -lam[k] * U[r * 3 + k])));
      rr = fma(v, v, rr);
    }
    const double excess = fma(U[k], U[k], fma(U[3 + k], U[3 + k], fma(U[6 + k], U[6 + k], -1.0)));
    ok &= rr <= kResidualTol * kResidualTol * nA && fabs(excess) <= kResidualTol;
  }
  return !ok;
}

// FP64 refinement of one flagged lane (compensated form): the arrow and the
// FP32 roots f[0..8] = (a1, a2, b1, b2, g, c, s, mu, nu), code = e << 2 | cls.
// A final FP64 Newton step on mu and nu (Sec. 1.4.2), eigenvectors re-formed
// in FP64; with `rec` (the input record), the FP64 residual check
// ||A u - lambda u|| <= 16 eps32 ||A||_F, whose failure is returned.
__device__ __forceinline__ bool refine_one(const float f[9], const int code, const float* rec, double lam[3],
                                        double U[9]) {
  f64::Lane D;
  D.a1 = f[0]; D.a2 = f[1]; D.b1 = f[2]; D.b2 = f[3]; D.g = f[4]; D.c = f[5]; D.s = f[6];
  D.cls = code & 3;
  D.e = code >> 2;
  double mu = f[7], nu = f[8];
  if (D.cls == kRed) {
    const double ab = D.a1 - D.a2, bb1 = D.b1 * D.b1, bb2 = D.b2 * D.b2;
    const double rab = rcp64(ab);
    const double g0 = D.g - D.a1, g1 = D.a2 - D.g;
    const double c0 = bb2 * rab, c1 = bb1 * rab;
    if (mu > 0.0) mu = f64::newton64(ab, bb1, bb2, g0, c0, -g0 - c0, mu);
    if (nu > 0.0) nu = f64::newton64(ab, bb2, bb1, g1, c1, -g1 - c1, nu);
  }
  f64::finish_lane(D, mu, nu, lam, U);
  return rec != nullptr && residual_fails(rec, lam, U);
}

// The refinement of one flagged matrix from its input record: in 62-bit fixed
// point (solve_fx.cuh; about 2600 issue slots a warp, the FP64 pipe needs 8600
// cycles) when its entries are of similar size, else refine_one on its FP32
// arrow and roots, formed again by the FP32 solve's own steps.  out:
// eigenvalues, then eigenvectors.  Whole warps call it; a lane without work
// passes active = false.  Not inlined: all kernels then share its code and
// return the same bits.  In the kernels that call it at their end (80 registers
// a thread) it and the call need 500 bytes of stack and spill some 350, per
// refined matrix only: more registers would leave fewer CTAs for the FP32 solve
// (5 per SM instead of 6: slower over all).
__device__ __noinline__ bool refine_record(const float* rec, const bool active, const bool check, float out[12]) {
  double lam[3], U[9];
  int rk[3] = {0, 1, 2};
  bool done = false, bad = false;
  if (active) {
    double a[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) a[k] = f2d_exact(rec[k]);
    const fx::Fixed F = fx::fixed_of<false>(a);
    if (F.similar && !F.diagonal && fx::solve<true, false>(F, nullptr, lam, U, rk)) {
      done = true;
      bad = check && residual_fails(rec, lam, U);
    }
  }
  if (__any_sync(0xffffffffu, active && !done)) {
    Lane32 L;
    L.cls = kIdle;
    if (active && !done) L = make_lane32<true>(rec);
    float root[2];
    roots_of<true>(L, root);
    if (active && !done) {
      const float f[9] = {L.a1, L.a2, L.b1, L.b2, L.g, L.c, L.s, root[0], root[1]};
      bad = refine_one(f, (L.e << 2) | L.cls, check ? rec : nullptr, lam, U);
      rk[0] = 0; rk[1] = 1; rk[2] = 2;
    }
  }
  if (active) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      out[rk[k]] = d2f_rn(lam[k]);
      // The sign rule holds for the rounded components (two may become equal).
      const float y0 = d2f_rn(U[k]), y1 = d2f_rn(U[3 + k]), y2 = d2f_rn(U[6 + k]);
      const unsigned sb = sign_of_largest(y0, y1, y2);
      out[3 + rk[k]] = __uint_as_float(__float_as_uint(y0) ^ sb);
      out[6 + rk[k]] = __uint_as_float(__float_as_uint(y1) ^ sb);
      out[9 + rk[k]] = __uint_as_float(__float_as_uint(y2) ^ sb);
    }
  }
  return bad;
}

// Rows of a CTA's flagged matrices, refined after its last tile (or when a
// further tile might not fit).
template <bool kServe>
struct FlagList;
template <>
struct FlagList<false> {
  static constexpr int kCap = 1024;
  uint32_t seq[kCap];  // place in the CTA's sequence of tiles x tile size + row
};
template <>
struct FlagList<true> {
  static constexpr int kCap = 512;
  TileRef<float> at[kCap];  // the row's record and outputs
};

// kMode: kPlain (SYEV3_F32), kComp32 (compensated: the flagged matrices are
// listed, and refined by the CTA's whole warps at the end) or kDeferred
// (compensated: they are appended to a list in the caller's workspace, for
// k_refine_list).  Refining at the end, the SM's warps run in step, which
// matters for 40 KB of straight-line code: with 4 % of 2^22 matrices flagged
// kComp32 took 219 us (191 with the present zero finder); refined by single
// warps as soon as 32 had gathered, 295; by FP64 code on a list per tile (the
// earlier form) 281.
// kVectors = false (plain mode only): eigenvalues only, U_out NULL.
// kRows: matrices per thread and tile.
// kServe: the serving build.  The tiles are those of the
// device-resident work list `list` (A, n, lam_out and U_out are unused), each
// with its own input and output rows; a tile's input is bulk-copied from its
// first 16-byte boundary-aligned record on, or loaded with plain loads when
// its start is not 16-byte aligned.  The production builds (kServe = false)
// compile this out.
template <bool kBulkIn, int kMode, bool kVectors = true, bool kServe = false, int kRows = 1>
__global__ void __launch_bounds__(kTPB, kMode == kPlain ? 11 : (kMode == kComp32 ? 6 : 8))
    k_syev3_f32(const float* __restrict__ A, int64_t n, float* __restrict__ lam_out, float* __restrict__ U_out,
                unsigned long long* __restrict__ counters, int64_t* __restrict__ flag_list,
                unsigned long long* __restrict__ flag_count, const ServeList* __restrict__ list) {
  static_assert(!kServe || (kBulkIn && kMode != kDeferred && kVectors), "the serving build is bulk, vectors");
  static_assert(kTPB == kServeTile, "serving tiles are solve tiles");
  static_assert(kRows == 1 || (kMode == kPlain && !kServe), "longer tiles: production, plain");
  constexpr bool kComp = kMode != kPlain, kList = kMode == kComp32;
  constexpr int kTile = kTPB * kRows;
  __shared__ alignas(16) float s_in[2][kTile * 6];
  __shared__ alignas(16) float s_lam[kTile * 3];
  __shared__ alignas(16) float s_U[kTile * 9];
  __shared__ alignas(8) uint64_t s_bar[2];
  __shared__ TileRef<float> s_ref[kServe ? 2 : 1];  // serving build: the tile of each buffer
  constexpr int kCap = FlagList<kServe>::kCap;
  __shared__ std::conditional_t<kList, FlagList<kServe>, int> s_list;
  __shared__ int s_nflag;

  const int tid = threadIdx.x, lane_id = tid & 31;
  const int64_t n_tiles = kServe ? list->n_tiles : (n + kTile - 1) / kTile;
  bool want_U = (U_out != nullptr);
  bool vec_lam = ((reinterpret_cast<uintptr_t>(lam_out) & 15) == 0);
  bool vec_U = want_U && ((reinterpret_cast<uintptr_t>(U_out) & 15) == 0);
  int64_t cursor = 0;  // serving build: item cursor of the tiles this CTA issues (thread 0)

  if (tid == 0) {
    s_nflag = 0;
    if (kBulkIn) {
      mbar_init(&s_bar[0], 1);
      mbar_init(&s_bar[1], 1);
      fence_mbar_init();
    }
  }
  __syncthreads();

  // Bulk-copy part of a tile: its first (cnt * 24) & ~15 bytes; the odd last
  // record of a tile with an odd count (8 bytes past a 16-byte boundary) is
  // loaded with plain loads after the wait.
  auto issue = [&](int64_t tile, int buf) {
    if constexpr (kServe) {
      const TileRef<float> r = serve_tile<float>(list, tile, cursor);
      s_ref[buf] = r;
      const uint32_t bytes = (reinterpret_cast<uintptr_t>(r.src) & 15) ? 0u : (((uint32_t)r.cnt * 24u) & ~15u);
      if (bytes == 0) {  // plain loads after the wait
        mbar_arrive(&s_bar[buf]);
        return;
      }
      mbar_arrive_expect_tx(&s_bar[buf], bytes);
      bulk_g2s(s_in[buf], r.src, bytes, &s_bar[buf]);
      return;
    }
    const int64_t base = tile * kTile;
    const int cnt = (int)((n - base) < kTile ? (n - base) : kTile);
    const uint32_t bytes = ((uint32_t)cnt * 24u) & ~15u;
    mbar_arrive_expect_tx(&s_bar[buf], bytes);
    if (bytes) bulk_g2s(s_in[buf], A + base * 6, bytes, &s_bar[buf]);
  };

  // Refines the listed matrices; every thread of the CTA calls it.
  auto refine = [&]() {
    if (tid == 0) bulk_write_wait();  // the FP32 results are in memory
    __syncthreads();
    const int count = s_nflag;
    if constexpr (kList) {
      for (int i0 = tid & ~31; i0 < count; i0 += kTPB) {  // whole warps
        const bool active = i0 + lane_id < count;
        float rec[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, out[12];
        float *dl = nullptr, *dU = nullptr;
        if (active) {
          const float* src;
          if constexpr (kServe) {
            const TileRef<float> r = s_list.at[i0 + lane_id];
            src = r.src;
            dl = r.lam;
            dU = r.U;
          } else {
            const uint32_t q = s_list.seq[i0 + lane_id];
            const int64_t row = ((int64_t)(q / kTPB) * gridDim.x + blockIdx.x) * kTPB + q % kTPB;
            src = A + row * 6;
            dl = lam_out + row * 3;
            dU = U_out ? U_out + row * 9 : nullptr;
          }
#pragma unroll
          for (int k = 0; k < 6; ++k) rec[k] = src[k];
        }
        const bool bad = refine_record(rec, active, counters != nullptr, out);
        if (bad) atomicAdd(&counters[3], 1ull);
        if (active) {
#pragma unroll
          for (int k = 0; k < 3; ++k) dl[k] = out[k];
          if (dU != nullptr) {
#pragma unroll
            for (int k = 0; k < 9; ++k) dU[k] = out[3 + k];
          }
        }
      }
    }
    __syncthreads();
    if (tid == 0) s_nflag = 0;
  };

  uint32_t phases = 0u;
  uint32_t seq = (uint32_t)tid;  // this thread's row in the CTA's sequence of tiles
  int buf = 0;
  int64_t tile = blockIdx.x;
  if (kBulkIn && tid == 0 && tile < n_tiles) issue(tile, 0);

  for (; tile < n_tiles; tile += gridDim.x, buf ^= 1, seq += kTPB) {
    const int64_t base = tile * kTile;
    int cnt = (int)((n - base) < kTile ? (n - base) : kTile);
    float* lam_tile = lam_out + base * 3;
    float* U_tile = want_U ? U_out + base * 9 : nullptr;
    const int64_t next = tile + gridDim.x;
    if (tid == 0) bulk_read_wait();  // the last tile's rows have left the staging area
    if (kBulkIn) {
      if (tid == 0 && next < n_tiles) issue(next, buf ^ 1);
      const bool ok = mbar_wait(&s_bar[buf], (phases >> buf) & 1u);
      if (__syncthreads_or(!ok)) {
        if (tid == 0) atomicOr(&g_flags32, kFlagWaitTimeout);
        mbar_wait(&s_bar[buf], (phases >> buf) & 1u);
        if (next < n_tiles) mbar_wait(&s_bar[buf ^ 1], (phases >> (buf ^ 1)) & 1u);
        return;
      }
      phases ^= 1u << buf;
      const float* src = A + base * 6;
      int done_f = (int)((((uint32_t)cnt * 24u) & ~15u) / 4u);
      if constexpr (kServe) {
        const TileRef<float> r = s_ref[buf];
        cnt = r.cnt;
        src = r.src;
        lam_tile = r.lam;
        U_tile = r.U;
        want_U = (r.U != nullptr);
        vec_lam = ((reinterpret_cast<uintptr_t>(r.lam) & 15) == 0);
        vec_U = want_U && ((reinterpret_cast<uintptr_t>(r.U) & 15) == 0);
        done_f = (reinterpret_cast<uintptr_t>(r.src) & 15) ? 0 : (int)((((uint32_t)cnt * 24u) & ~15u) / 4u);
      }
      if (done_f < cnt * 6) {
        for (int i = done_f + tid; i < cnt * 6; i += kTPB) s_in[buf][i] = src[i];
        __syncthreads();
      }
    } else {
      __syncthreads();  // the previous tile's records and staging have been read
      for (int i = tid; i < cnt * 6; i += kTPB) s_in[buf][i] = A[base * 6 + i];
      __syncthreads();
    }

    // (not unrolled: two copies of the solve would not fit the instruction cache)
#pragma unroll 1
    for (int row = tid; row < kTile; row += kTPB) {
      Lane32 L;
      L.cls = kIdle;
      L.near_defl = false;
      if (row < cnt) {
        const float2* src = reinterpret_cast<const float2*>(&s_in[buf][row * 6]);
        const float2 p0 = src[0], p1 = src[1], p2 = src[2];
        const float a_in[6] = {p0.x, p0.y, p1.x, p1.y, p2.x, p2.y};
        L = make_lane32<kComp>(a_in);
      }
      // The warp's lanes that form eigenpairs (taken where all 32 are together),
      // which rejoin after the class-specific part of the solve.
      const unsigned fin_mask = __ballot_sync(0xffffffffu, L.cls != kIdle && L.cls != kNonFin);
      float root[2];
      const bool capped = roots_of<kComp>(L, root);

      bool flagged = false, nonfinite = false;
      int rk[3] = {0, 1, 2};  // rank of each eigenpair (ascending); identity for the other paths
      if (L.cls != kIdle) {
        float l[3], U[9];
        if (L.cls == kNonFin) {
          nonfinite = true;
          const float qnan = __int_as_float(0x7fc00000);
#pragma unroll
          for (int k = 0; k < 3; ++k) l[k] = qnan;
#pragma unroll
          for (int k = 0; k < 9; ++k) U[k] = qnan;
        } else if (!kVectors) {
          finish32_values(L, root[0], root[1], l, fin_mask);
          unscale3(l, L.e);
        } else {
          finish32(L, root[0], root[1], l, U, rk, fin_mask);
          if (kComp && L.cls != kDiag) {
            // the eigenvalues' gaps in ascending order (min, median, max)
            const float lo = fminf(fminf(l[0], l[1]), l[2]), hi = fmaxf(fmaxf(l[0], l[1]), l[2]);
            const float md = fmaxf(fminf(l[0], l[1]), fminf(fmaxf(l[0], l[1]), l[2]));
            const float nrm2 = fmaf(lo, lo, fmaf(md, md, hi * hi));
            const float gap = fminf(md - lo, hi - md);
            flagged = capped || L.near_defl || (gap * gap < (kClusterTau * kClusterTau) * nrm2);
          }
          unscale3(l, L.e);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) s_lam[row * 3 + rk[k]] = l[k];
        if (kVectors) {
#pragma unroll
          for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int i = 0; i < 3; ++i) s_U[row * 9 + i * 3 + rk[k]] = U[i * 3 + k];
        }
      }

      if constexpr (kComp) {
        const unsigned m = __ballot_sync(0xffffffffu, flagged);
        const int before = __popc(m & ((1u << lane_id) - 1u));
        if constexpr (kList) {
          int at = 0;
          if (lane_id == 0 && m) at = atomicAdd(&s_nflag, __popc(m));
          at = __shfl_sync(0xffffffffu, at, 0) + before;
          if (flagged) {
            if constexpr (kServe)
              s_list.at[at] =
                  TileRef<float>{s_ref[buf].src + tid * 6, lam_tile + tid * 3, want_U ? U_tile + tid * 9 : nullptr, 1};
            else
              s_list.seq[at] = seq;
          }
        } else {
          unsigned long long at = 0;
          if (lane_id == 0 && m) at = atomicAdd(flag_count, (unsigned long long)__popc(m));
          at = __shfl_sync(0xffffffffu, at, 0);
          if (flagged) flag_list[at + before] = base + tid;
        }
      }
      if (counters != nullptr) {
        const unsigned cm = __ballot_sync(0xffffffffu, capped);
        const unsigned nf = __ballot_sync(0xffffffffu, nonfinite);
        const unsigned fl = __ballot_sync(0xffffffffu, flagged);
        if (lane_id == 0) {
          if (cm) atomicAdd(&counters[0], (unsigned long long)__popc(cm));
          if (nf) atomicAdd(&counters[1], (unsigned long long)__popc(nf));
          if (fl) atomicAdd(&counters[2], (unsigned long long)__popc(fl));
        }
      }
    }
    fence_async_shared();
    __syncthreads();

    // A full, aligned tile's rows leave by bulk copy; the staging area is
    // written again only after thread 0 has seen it read (above, before the
    // next tile's barrier).
    if (cnt == kTile && vec_lam && (!want_U || vec_U)) {
      if (tid == 0) {
        bulk_s2g(lam_tile, s_lam, kTile * 12);
        if (kVectors && want_U) bulk_s2g(U_tile, s_U, kTile * 36);
      }
    } else {
      auto store = [&](float* dst, const float* src, const int m, const bool vec) {
        const int m4 = vec ? m / 4 : 0;
        for (int i = tid; i < m4; i += kTPB)
          reinterpret_cast<float4*>(dst)[i] = reinterpret_cast<const float4*>(src)[i];
        for (int i = 4 * m4 + tid; i < m; i += kTPB) dst[i] = src[i];
      };
      store(lam_tile, s_lam, cnt * 3, vec_lam);
      if (kVectors && want_U) store(U_tile, s_U, cnt * 9, vec_U);
    }
    if constexpr (kList) {
      if (s_nflag > kCap - kTPB) refine();  // (s_nflag is stable between the tiles' barriers)
    }
  }
  if constexpr (kList) refine();
  if (tid == 0) bulk_read_wait();
}

// The refinement of the deferred form: the listed matrices, a CTA's warps in
// step (one barrier a turn): they share the fetches of the refinement's 40 KB
// of straight-line code, whose fetch is the main stall (the workspace form, 4 %
// flagged, 2^21 matrices 93.2 -> 90.0 us, 2^23 330.3 -> 327.7; CTAs of 256 and
// 512 threads: no better, slower).
__global__ void __launch_bounds__(kTPB, 5) k_refine_list(const int64_t* __restrict__ rows,
                                                         const unsigned long long* __restrict__ count,
                                                         const float* __restrict__ A, float* __restrict__ lam_out,
                                                         float* __restrict__ U_out,
                                                         unsigned long long* __restrict__ counters) {
  const int64_t m = (int64_t)*count;
  for (int64_t base = (int64_t)blockIdx.x * kTPB; base < m; base += (int64_t)gridDim.x * kTPB) {
    __syncthreads();
    const int64_t i = base + threadIdx.x;
    const bool active = i < m;
    const int64_t row = rows[active ? i : m - 1];
    float rec[6], out[12];
#pragma unroll
    for (int k = 0; k < 6; ++k) rec[k] = A[row * 6 + k];
    const bool bad = refine_record(rec, active, counters != nullptr, out);
    if (bad) atomicAdd(&counters[3], 1ull);
    if (active) {
#pragma unroll
      for (int k = 0; k < 3; ++k) lam_out[row * 3 + k] = out[k];
      if (U_out != nullptr) {
#pragma unroll
        for (int k = 0; k < 9; ++k) U_out[row * 9 + k] = out[3 + k];
      }
    }
  }
}

template <bool kBulkIn, int kMode, bool kVectors, bool kServe = false, int kRows = 1>
int blocks_per_sm_f32() {
  static int cached = -1;
  if (cached < 0) {
    int v = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &v, k_syev3_f32<kBulkIn, kMode, kVectors, kServe, kRows>, kTPB, 0);
    cached = (e == cudaSuccess && v > 0) ? v : 1;
  }
  return cached;
}

template <bool kBulkIn, int kMode, bool kVectors = true, int kRows = 1>
cudaError_t launch(const float* A, int64_t n, float* lam, float* U, unsigned long long* counters, cudaStream_t stream,
                   int sms, int64_t* flag_list = nullptr, unsigned long long* flag_count = nullptr) {
  constexpr int kTile = kTPB * kRows;
  const int64_t n_tiles = (n + kTile - 1) / kTile;
  const int64_t resident = (int64_t)sms * blocks_per_sm_f32<kBulkIn, kMode, kVectors, false, kRows>();
  const int grid = (int)(n_tiles < resident ? n_tiles : resident);
  k_syev3_f32<kBulkIn, kMode, kVectors, false, kRows>
      <<<grid, kTPB, 0, stream>>>(A, n, lam, U, counters, flag_list, flag_count, nullptr);
  return cudaGetLastError();
}

template <int kMode>
cudaError_t launch_serve(const ServeList* list, unsigned long long* counters, cudaStream_t stream, int sms) {
  // The list's length is known only on the device: a resident grid; CTAs
  // without a tile exit at once.
  const int grid = sms * blocks_per_sm_f32<true, kMode, true, true>();
  k_syev3_f32<true, kMode, true, true><<<grid, kTPB, 0, stream>>>(nullptr, 0, nullptr, nullptr, counters, nullptr, nullptr, list);
  return cudaGetLastError();
}

}  // namespace

// From these sizes on the plain kernel takes two matrices per thread and tile:
// half the barriers, waits and loop overhead per matrix, against fewer tiles
// than keep every CTA busy to the end.  us, two rows against one: eigenvalues
// only (tensors) 2^23 127 / 139, 2^20 17.7 / 19.4, 2^19 9.8 / 10.4, 300763
// 7.1 / 6.6; with eigenvectors (mixed), whose tiles then cost shared memory for
// 9 CTAs per SM instead of 12, 2^23 174.5 / 177.0, 3000001 64.4 / 65.3, 2^21
// 46.8 / 47.0, 2^20 24.6 / 24.2.
constexpr int64_t kTwoRowsValues = (int64_t)1 << 19, kTwoRowsVectors = (int64_t)1 << 21;

cudaError_t launch_f32(const float* A, int64_t n, float* lam, float* U, bool compensated,
                       unsigned long long* counters, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const bool bulk = (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  if (compensated)
    return bulk ? launch<true, kComp32>(A, n, lam, U, counters, stream, sms)
                : launch<false, kComp32>(A, n, lam, U, counters, stream, sms);
  if (bulk && U == nullptr)
    return n >= kTwoRowsValues ? launch<true, kPlain, false, 2>(A, n, lam, U, counters, stream, sms)
                            : launch<true, kPlain, false>(A, n, lam, U, counters, stream, sms);
  if (bulk && n >= kTwoRowsVectors) return launch<true, kPlain, true, 2>(A, n, lam, U, counters, stream, sms);
  return bulk ? launch<true, kPlain>(A, n, lam, U, counters, stream, sms)
              : launch<false, kPlain>(A, n, lam, U, counters, stream, sms);
}

// From this size on the workspace form lists its flagged matrices there and
// refines them with a second kernel: the solve then needs 56 registers instead
// of 80 (9 CTAs per SM instead of 6), which pays for the second launch and the
// list.  Measured, us, this form against the single kernel: 2^23 matrices with
// 4 % flagged 328 / 370, 2^21 90 / 101; when the line was drawn 2^21 97 / 114
// with 4 % flagged and 76 / 72 with none, 2^20 58 / 68 and 45 / 42.  (The
// earlier form, the refinement by FP64 code on a second stream beside the
// solve: 414 at 2^23.)
constexpr int64_t kDeferMin = (int64_t)1 << 21;

cudaError_t launch_f32c_ws(const float* A, int64_t n, float* lam, float* U, unsigned long long* counters, void* work,
                           cudaStream_t stream) {
  if (n < kDeferMin) return launch_f32(A, n, lam, U, true, counters, stream);
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  auto* count = static_cast<unsigned long long*>(work);
  auto* rows = reinterpret_cast<int64_t*>(static_cast<char*>(work) + kFlagListOffset);
  e = cudaMemsetAsync(count, 0, sizeof(*count), stream);
  if (e != cudaSuccess) return e;
  e = (reinterpret_cast<uintptr_t>(A) & 15) == 0
          ? launch<true, kDeferred>(A, n, lam, U, counters, stream, sms, rows, count)
          : launch<false, kDeferred>(A, n, lam, U, counters, stream, sms, rows, count);
  if (e != cudaSuccess) return e;
  k_refine_list<<<sms * 5, kTPB, 0, stream>>>(rows, count, A, lam, U, counters);
  return cudaGetLastError();
}

cudaError_t launch_f32_serve(const ServeList* list, bool compensated, unsigned long long* counters,
                             cudaStream_t stream) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  return compensated ? launch_serve<kComp32>(list, counters, stream, sms)
                     : launch_serve<kPlain>(list, counters, stream, sms);
}

cudaError_t take_flags_f32(unsigned* flags) {
  unsigned v = 0, zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, g_flags32, sizeof(v));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(g_flags32, &zero, sizeof(zero));
  *flags |= v;
  return e;
}

}  // namespace syev3
