// fmb_cam.cuh -- the camera-plane form of a ray/Gaussian pair that the two-parameter
// render and its adjoint evaluate, and the per (view, Gaussian) records it reads.
//
// A pixel's ray is c = ((px - cx)/fx, (py - cy)/fy, 1): affine in the pixel.  In the
// camera frame the precision is P = A A^T with A = R L, and any root of it serves,
// since Eq. 2 depends on L only through P.  The lower Cholesky factor B of P makes
// the whitened ray a = B^T c as short as it gets: a2 is constant, a1 depends on py
// only.  With m the mean in the camera frame (z its depth) and c_e a fixed pixel near
// the mean's projection, write c = c_e + delta and measure the hit from the mean's
// own depth: t = z + tau.  Then
//   D   = z B^T delta - B^T (m - z c_e)      (affine in the pixel, third entry 0)
//   tau = -(D . a) / (a . a),   u = D + tau a,   q = u . u
// The pixel offsets from c_e are exact near the projection (Sterbenz) and m - z c_e
// is formed in float pairs, so u keeps its relative accuracy for rays that pass close
// to a distant mean, where t a - b in plain fp32 loses |b|/|u| ulps.  25 operations
// per pair without the normal, 36 with it (42 for flat Gaussians, cam_flat_flags); the world-frame evaluation (exact float
// pairs of the ray and of mu - o, and a second projection of u) took 35 and 56 at the
// same error (log-weights 1.0-2.1e-6 rms against 1.3-2.2e-6, FP64 comparison on the
// benchmark's scenes).
//
// Every whitened quantity carries a factor sqrt(log2(e) / 2), so that
// u . u - log2(lambda) is -log2(delta) of Eq. 4, and lengths are in pixels (B's rows
// divided by fx, fy), so that the pixel offsets enter as they are.
#pragma once

#include "fmb_f32x2.cuh"
#include "fmb_internal.cuh"

namespace fmb {

// Record of two Gaussians (one per packed lane), 16 f2 = 128 bytes.  B' = [[B00],
// [B10, B11], [e0, e1, e2]] is the root in the frame of the offsets (dx, dy, 1).
//   0 -pe_x  1 -pe_y   expansion pixel, negated
//   2 B00  3 B10  4 z  5 d0  6 e0  7 B11  8 e1  9 z B11  10 d1
//   11 e2^2  12 -log2(lambda)  13 flags (bits)  14 rho_x  15 rho_y (m - z c_e, in pixels)
// An object's last record of an odd count holds its last Gaussian twice, the copy
// with the log-density -1e30, so that its density is exactly 0, and flagged
// kCamCopy: the forward leaves its weight out.  (Its weight's exponent passes through
// beta1, which may be 0 or negative.  The adjoint's sums of its lane are not read.)
// kCamFlat, kCamFlatter: see cam_flat_flags.
constexpr int kCamF2 = 16;
constexpr float kDummyNl2 = 1e30f;
constexpr int kCamFlat = 1, kCamCopy = 2, kCamFlatter = 4;

// The rounding of tau leaves a component dtau a in u, to which u . u is stationary but
// the normal g = B u is not: it moves by dtau P c, and |P c| exceeds |g| by up to the
// square of the axis ratio.  A second projection of u onto the complement of a (6
// operations) takes it out.  Only flat Gaussians need it.  With l1 >= l2 >= l3 the axes
// of the root, tr(P)^2 over the sum of P's principal 2x2 minors is about (l1/l2)^2 / 2
// (thin discs) and tr(P) tr(P^-1) about 2 (l1/l3)^2 (needles too).  Normals of discs
// (sigma 0.4, depth 4, rms against FP64; projected / not): ratio 3 0.8e-7 / 0.7e-7, 6 1.1e-7 /
// 2.0e-7, 10 1.4e-7 / 5.1e-7, 30 1.7e-7 / 4.4e-6, 100 1.7e-7 / 4.9e-5, growing with the square:
// the forward projects from a ratio of 5 on (4 % of the benchmark's Gaussians).  The
// gradients were within the projected form's up to a ratio of 30 (L: 1.1e-5 / 1.8e-5) and
// past it at 100 (1.2e-4 / 0.9e-5): the adjoint, whose warps hold 64 Gaussians each, projects
// from 16 on.  Both rules cost the benchmark's scenes at most 0.3 % (orbit 648.6 ->
// 650.8 us; 1023x767 at K = 333 358 before, 357 with one flagged record at a time); a scene of
// discs of ratio 20 14 % forward and 4 % in the adjoint.
__device__ __forceinline__ int cam_flat_flags(float trace, float minors, float det) {
  const bool needle = !(trace * minors < 1000.f * det);
  return (needle || !(trace * trace < 14.f * minors) ? kCamFlat : 0) |
         (needle || !(trace * trace < 130.f * minors) ? kCamFlatter : 0);
}

// sqrt(log2(e) / 2), its square, and 2 ln 2 (the derivative of d = ln(delta) with
// respect to a scaled u is -2 ln 2 u).
constexpr float kCamScale = 0.84932180028801904f;
constexpr float kCamScale2 = 0.72134752044448170f;
constexpr float kTwoLn2 = 1.3862943611198906f;

// Float pairs (unevaluated sums h + l, about 2^-46 relative): the prologue of the
// camera-plane records forms P = A A^T and its Cholesky factor in them, since P
// squares the condition of L, and the adjoint solves for a flat Gaussian's gradients.
// About 900 fp32 instructions per record; FP64 would take fewer, but issues one warp
// instruction per 16 cycles and SM here.
struct FF {
  float h, l;
};
__device__ __forceinline__ FF ff_renorm(float h, float l) {
  const float s = __fadd_rn(h, l);
  return FF{s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ FF operator+(FF a, FF b) {
  float s, e;
  two_sum(a.h, b.h, s, e);
  return ff_renorm(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ FF operator-(FF a) { return FF{-a.h, -a.l}; }
__device__ __forceinline__ FF operator-(FF a, FF b) { return a + (-b); }
__device__ __forceinline__ FF operator*(FF a, FF b) {
  float p, e;
  two_prod(a.h, b.h, p, e);
  return ff_renorm(p, fmaf(a.h, b.l, fmaf(a.l, b.h, e)));
}
__device__ __forceinline__ FF operator*(FF a, float b) {
  float p, e;
  two_prod(a.h, b, p, e);
  return ff_renorm(p, fmaf(a.l, b, e));
}
__device__ __forceinline__ FF ff_prod(float a, float b) {
  FF r;
  two_prod(a, b, r.h, r.l);
  return r;
}
__device__ __forceinline__ FF ff_diff(float a, float b) {
  FF r;
  two_sum(a, -b, r.h, r.l);
  return r;
}
// 1 / a and 1 / sqrt(a): one Newton step in pair arithmetic from the fp32 value.
__device__ __forceinline__ FF ff_rcp(FF a) {
  const float y = __frcp_rn(a.h);
  const FF r = FF{1.f, 0.f} - a * y;
  return ff_renorm(y, __fmul_rn(y, r.h));
}
__device__ __forceinline__ FF ff_rsqrt(FF a) {  // 0 for a <= 0 (a singular precision)
  if (!(a.h > 0.f)) return FF{a.h == a.h ? 0.f : a.h, 0.f};
  const float y = rsqrtf(a.h);
  const FF r = FF{1.f, 0.f} - a * ff_prod(y, y);
  return ff_renorm(y, __fmul_rn(0.5f * y, r.h));
}

struct CamRec2 {
  f2 npx, npy, B00, B10, z, d0, e0, B11, e1, F11, d1, ee, nl2;
  unsigned long long flags;  // of the two Gaussians, one per half
};
__device__ __forceinline__ CamRec2 cam_load(const ulonglong2* __restrict__ r) {
  const ulonglong2 q0 = r[0], q1 = r[1], q2 = r[2], q3 = r[3], q4 = r[4], q5 = r[5], q6 = r[6];
  CamRec2 g;
  g.npx = as_f2(q0.x);
  g.npy = as_f2(q0.y);
  g.B00 = as_f2(q1.x);
  g.B10 = as_f2(q1.y);
  g.z = as_f2(q2.x);
  g.d0 = as_f2(q2.y);
  g.e0 = as_f2(q3.x);
  g.B11 = as_f2(q3.y);
  g.e1 = as_f2(q4.x);
  g.F11 = as_f2(q4.y);
  g.d1 = as_f2(q5.x);
  g.ee = as_f2(q5.y);
  g.nl2 = as_f2(q6.x);
  g.flags = q6.y;
  return g;
}

// One pair per lane: two Gaussians against the pixel (X, Y), both lanes alike.
struct CamGeom2 {
  f2 dx, dy, a0, a1, ninv, tau, t, u0, u1, nx;  // ninv = -1 / a.a;  nx = -log2(delta)
};
__device__ __forceinline__ f2 rcp_neg_2(f2 a) { return pk(rcp_approx(-lo(a)), rcp_approx(-hi(a))); }
// The second projection of u (see cam_flat_flags).
__device__ __forceinline__ void cam_project2(CamGeom2& G, const CamRec2& g) {
  const f2 nk = mul2(fma2(G.u0, G.a0, fma2(G.u1, G.a1, mul2(G.tau, g.ee))), G.ninv);
  G.u0 = fma2(nk, G.a0, G.u0);
  G.u1 = fma2(nk, G.a1, G.u1);
}
template <bool PROJECT = false>
__device__ __forceinline__ CamGeom2 cam_geom2(const CamRec2& g, f2 X, f2 Y) {
  CamGeom2 G;
  G.dx = add2(X, g.npx);
  G.dy = add2(Y, g.npy);
  const f2 ad = fma2(g.B00, G.dx, mul2(g.B10, G.dy));
  G.a0 = add2(ad, g.e0);
  G.a1 = fma2(g.B11, G.dy, g.e1);
  const f2 D0 = fma2(g.z, ad, g.d0);
  const f2 D1 = fma2(g.F11, G.dy, g.d1);
  const f2 aa = fma2(G.a0, G.a0, fma2(G.a1, G.a1, g.ee));
  G.ninv = rcp_neg_2(aa);
  G.tau = mul2(fma2(D0, G.a0, mul2(D1, G.a1)), G.ninv);
  G.t = add2(g.z, G.tau);
  G.u0 = fma2(G.tau, G.a0, D0);
  G.u1 = fma2(G.tau, G.a1, D1);
  G.nx = fma2(G.u0, G.u0, fma2(G.u1, G.u1, fma2(mul2(G.tau, G.tau), g.ee, g.nl2)));
  if (PROJECT) cam_project2(G, g);
  return G;
}

// Reciprocal, reciprocal square root and square root to about an ulp from the MUFU
// approximation and one Newton step (3 to 5 instructions; the IEEE forms take 10 to 20,
// and the per-ray code of K = 100 was a quarter of the forward's instructions with
// them).  For normal, positive, finite arguments (0 and infinity give NaN); explicitly rounded, so that the forward and
// the adjoint (compiled with different flags) get the same bits.
__device__ __forceinline__ float rcp_nr(float x) {
  const float r = rcp_approx(x);
  return __fmaf_rn(r, __fmaf_rn(-x, r, 1.0f), r);
}
__device__ __forceinline__ float rsqrt_nr(float x) {
  const float r = rsqrt_approx(x);
  return __fmaf_rn(__fmul_rn(0.5f, r), __fmaf_rn(-__fmul_rn(x, r), r, 1.0f), r);
}
__device__ __forceinline__ float sqrt_nr(float x, float rsqrt_x) {
  const float s = __fmul_rn(x, rsqrt_x);
  return __fmaf_rn(__fmul_rn(0.5f, rsqrt_x), __fmaf_rn(-s, s, x), s);
}

// Camera-plane quantities of a pixel: its centre (px, py), c = (x, y, 1), |c| and its
// reciprocal.
struct CamRay {
  float px, py, x, y, len, ilen;
};
__device__ __forceinline__ CamRay cam_ray_at(const DevView& V, float px, float py) {
  CamRay r;
  r.px = px;
  r.py = py;
  r.x = __fmul_rn(__fsub_rn(px, V.cx), rcp_nr(V.fx));
  r.y = __fmul_rn(__fsub_rn(py, V.cy), rcp_nr(V.fy));
  const float cc = __fmaf_rn(r.x, r.x, __fmaf_rn(r.y, r.y, 1.0f));
  r.ilen = rsqrt_nr(cc);
  r.len = sqrt_nr(cc, r.ilen);
  return r;
}
__device__ __forceinline__ CamRay cam_ray(const DevView& V, int p) {
  const int iy = p / V.W;
  return cam_ray_at(V, static_cast<float>(p - iy * V.W) + 0.5f, static_cast<float>(iy) + 0.5f);
}

}  // namespace fmb
