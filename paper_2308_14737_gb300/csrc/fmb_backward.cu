// fmb_backward.cu -- adjoint of the forward render (the derivative of Eq. 2, 3, 4,
// 7, 8, 17 and of the Sec. 5 flow) with respect to the means, the precision
// factors L, the weights lambda and the camera poses.
//
// Layout of the work: a CTA takes one view, one tile of rays and one block of
// Gaussians.  Phase 1 turns each ray's upstream gradients into a record in shared
// memory (the per-pixel part of the adjoint: flow, normal renormalisation, alpha),
// every value stored twice so that one 16-byte load yields two broadcast pairs.
// When every view runs as two Gaussian blocks, grid mode launches the two CTAs of
// a ray tile as one 2-CTA cluster: each builds half of the tile's records and
// writes them into both CTAs' shared memory (distributed shared memory), so the
// per-ray work is done once per ray instead of once per block.
// Phase 2 is Gaussian-parallel: each thread owns two Gaussians, one per lane of
// packed FP32x2 arithmetic, recomputes their pair terms for every ray of its
// subgroup from the saved log-normaliser (no per-pair state was stored by the
// forward) and accumulates both Gaussians' gradient sums in registers.  Phase 3 combines the subgroups, converts the sums
// into gradients of mu, L, lambda and of the pose, and writes them once per CTA
// (fp32 atomics, or per-CTA partials that a second kernel adds in a fixed order).
//
// Adjoint in the camera-plane form of fmb_cam.cuh (a = B^T c, D = B^T d3 with
// d3 = z c - m, t = z + tau, u = D + tau a, g = B u, n = g/|g|, what = softmax of e):
//   ebar  = what (Dbar (t - D) + Nbar . n)            (softmax of Eq. 3)
//   dbar  = beta1 ebar + Abar e^{-sum delta} delta     (Eq. 7, Eq. 8)
//   gbar  = what/|g| (Nbar - (n . Nbar) n)             (Eq. 17 normalisation)
//   tbar  = Dbar what - (beta2/eta) ebar + (B^T gbar) . a
//   ubar  = B^T gbar - dbar u,   s = -tbar / a.a
//   y     = Dbar_vec = ubar + s a,   abar = tau y + s u
// (the contribution -dbar u.a of tbar is dropped: u . a = 0 exactly at the
// max-likelihood depth).  Since n is perpendicular to c and B is triangular, gbar
// needs the first two components only, and u's third enters through
// sigma = s - dbar tau and kappa = tau (sigma + s) alone (abar_2 = kappa e2,
// y_2 = sigma e2).  The render depends on B only through P = B B^T, so the gradient
// with respect to a full 3x3 root is X B with X symmetric (X = 2 Pbar), and the six
// lower entries that are accumulated give X, and with it the three upper ones, by
// substitution; then with A = R L Lbar = lower(R^T (X B) (B^-1 A)) and Rbar =
// (X B) B^T R^-T, and the mean's gradient comes from sum y.  Ten sums per Gaussian instead of the nineteen of the world-frame form, and with
// normals and pose gradients five more (below).
#include <algorithm>

#include "fmb_cam.cuh"
#include "fmb_f32x2.cuh"
#include "fmb_internal.cuh"

namespace fmb {

constexpr int kBwdMaxThreads = 160;
// Resident CTAs per SM the register budget targets (128 registers; with 2, the orbit 498
// against 467 us, 20 views 640x480 at K = 256 3.12 against 3.02 ms).
constexpr int kBwdMinBlocks = 3;
// Pair-loop unrolling: independent rays the scheduler can interleave (orbit 449 / 459 /
// 454 us with 3 / 2 / 1, without normals 2.98 / 2.97 / 2.96 ms).
template <bool NORMALS>
constexpr int bwd_unroll() {
  return NORMALS ? 3 : 1;
}

// Per-thread gradient sums of the thread's two Gaussians (one per lane).  y, abar,
// B00 .. are scaled and in pixels as the records are (fmb_cam.cuh).
//   0 A00  1 A10  2 A11   sum dx p0 + gb0 u0, dy p0 + gb1 u0, dy p1 + gb1 u1 (p = t y + s u)
//   3 Y0   4 Y1   5 Sg    sum y, sum sigma
//   6 E0   7 E1   8 Kp    sum abar, sum kappa (abar from sum p - z sum y instead costs
//                         two operations less and three times the error of Lbar)
//   9 nd                  -2 ln 2 sum dbar
//   NORMALS with pose gradients: T00 T01 T11 V0 V1, sum over the pairs of
//     what (n . Nbar) n n^T / |g|^2 in the first two components, and of its products
//     with dx h0 + dy h1 (for the third)
//   COLOR: sum what Cbar (3)
constexpr int kAccBase = 10;
template <bool NORMALS, bool COLOR, bool POSE>
__host__ __device__ constexpr int acc_count() {
  return kAccBase + (NORMALS && POSE ? 5 : 0) + (COLOR ? 3 : 0);
}
template <bool NORMALS, bool COLOR, bool POSE>
struct BwdAcc2 {
  static constexpr int kN = acc_count<NORMALS, COLOR, POSE>();
  static constexpr int kT = kAccBase, kCol = kN - 3;
  f2 v[kN];
};

// Shared-memory record of one ray, every value duplicated so that one 16-byte load
// gives two broadcast pairs:
//   [X Y | -lse2 K2 | Dbar -D | -KA -B2E]
//   NORMALS: [Nt0 Nt1 | m00 m01 | m11 0]      COLOR: [Cb0 Cb1 | Cb2 -Cbar.C]
// X, Y: pixel centre.  K2 = -(beta2/eta) log2(e) |c|, B2E = (beta2/eta) |c|, Dbar the
// depth's upstream gradient times |c| (t is measured along z), D the depth along z
// (t - D is formed first: it is exact where one Gaussian is seen), KA = 2 ln 2 Abar
// e^-sum delta.  Nt = (fx (Nbar_0 - x Nbar_2), fy (Nbar_1 - y Nbar_2)): Nbar applied
// to the image-plane components h of g.  m: minus the quadratic form |g|^2 of h.
template <bool NORMALS, bool COLOR>
__host__ __device__ constexpr int ray_rec2() {
  return 4 + (NORMALS ? 3 : 0) + (COLOR ? 2 : 0);
}

// FLAT: a warp with flat Gaussians (cam_flat_flags); `flat` says so where one loop serves both.
template <bool NORMALS, bool COLOR, bool POSE, bool FLAT>
__device__ __forceinline__ void bwd_pair2(BwdAcc2<NORMALS, COLOR, POSE>& S, const CamRec2& g,
                                          const ulonglong2* __restrict__ rr, f2 nB1, f2 nB1s, f2 tiny, f2 c0,
                                          f2 c1, f2 c2, bool flat = false) {
  using Acc = BwdAcc2<NORMALS, COLOR, POSE>;
  const ulonglong2 q0 = rr[0], q1 = rr[1], q2 = rr[2], q3 = rr[3];
  const f2 nlse = as_f2(q1.x), K2 = as_f2(q1.y), Dbar = as_f2(q2.x), nD = as_f2(q2.y), nKA = as_f2(q3.x),
           nB2E = as_f2(q3.y);
  CamGeom2 G = cam_geom2<FLAT && NORMALS>(g, as_f2(q0.x), as_f2(q0.y));
  if (COLOR && NORMALS && flat) cam_project2(G, g);
  const f2 what = ex2_2(fma2(G.t, K2, fma2(G.nx, nB1, nlse)));
  const f2 delta = pk(ex2_approx(-lo(G.nx)), ex2_approx(-hi(G.nx)));
  const f2 Dw = mul2(Dbar, what), tD = add2(G.t, nD);
  f2 br;  // the bracket of ebar, unless it is the depth's term alone
  f2 rs, nN, h0, h1, m0, m1, Nt0, Nt1;
  if (NORMALS) {
    const ulonglong2 q4 = rr[4], q5 = rr[5], q6 = rr[6];
    Nt0 = as_f2(q4.x);
    Nt1 = as_f2(q4.y);
    h0 = mul2(g.B00, G.u0);
    h1 = fma2(g.B11, G.u1, mul2(g.B10, G.u0));
    m0 = fma2(as_f2(q5.y), h1, mul2(as_f2(q5.x), h0));  // minus the metric times h
    m1 = fma2(as_f2(q6.x), h1, mul2(as_f2(q5.y), h0));
    const f2 ngg = fma2(h0, m0, fma2(h1, m1, tiny));    // -|g|^2 (tiny < 0)
    rs = pk(rsqrt_approx(-lo(ngg)), rsqrt_approx(-hi(ngg)));
    nN = mul2(fma2(Nt0, h0, mul2(Nt1, h1)), rs);
    br = fma2(Dbar, tD, nN);
  }
  f2 Cb0, Cb1, Cb2;
  if (COLOR) {  // Cbar . c_i joins the weight's gradient (Eq. 3 with colours)
    const ulonglong2 q7 = rr[NORMALS ? 7 : 4], q8 = rr[NORMALS ? 8 : 5];
    Cb0 = as_f2(q7.x);
    Cb1 = as_f2(q7.y);
    Cb2 = as_f2(q8.x);
    const f2 cc = fma2(Cb2, c2, fma2(Cb1, c1, fma2(Cb0, c0, as_f2(q8.y))));
    br = NORMALS ? add2(br, cc) : fma2(Dbar, tD, cc);
  }
  const f2 ebar = NORMALS || COLOR ? mul2(what, br) : mul2(Dw, tD);
  const f2 nd = fma2(nB1s, ebar, mul2(nKA, delta));
  f2 tbar = fma2(nB2E, ebar, Dw);
  f2 ub0, ub1;
  if (!NORMALS) {
    ub0 = mul2(nd, G.u0);
    ub1 = mul2(nd, G.u1);
  } else {
    const f2 sc = mul2(what, rs);
    const f2 sN = mul2(mul2(sc, rs), nN);
    const f2 gb0 = fma2(sN, m0, mul2(sc, Nt0));
    const f2 gb1 = fma2(sN, m1, mul2(sc, Nt1));
    const f2 b0 = fma2(g.B10, gb1, mul2(g.B00, gb0));
    const f2 b1 = mul2(g.B11, gb1);
    tbar = fma2(b1, G.a1, fma2(b0, G.a0, tbar));
    ub0 = fma2(nd, G.u0, b0);
    ub1 = fma2(nd, G.u1, b1);
    S.v[0] = fma2(gb0, G.u0, S.v[0]);
    S.v[1] = fma2(gb1, G.u0, S.v[1]);
    S.v[2] = fma2(gb1, G.u1, S.v[2]);
    if (POSE) {
      const f2 r0 = mul2(sN, h0), r1 = mul2(sN, h1), w = fma2(G.dx, h0, mul2(G.dy, h1));
      S.v[Acc::kT + 0] = fma2(r0, h0, S.v[Acc::kT + 0]);
      S.v[Acc::kT + 1] = fma2(r0, h1, S.v[Acc::kT + 1]);
      S.v[Acc::kT + 2] = fma2(r1, h1, S.v[Acc::kT + 2]);
      S.v[Acc::kT + 3] = fma2(r0, w, S.v[Acc::kT + 3]);
      S.v[Acc::kT + 4] = fma2(r1, w, S.v[Acc::kT + 4]);
    }
  }
  const f2 s = mul2(tbar, G.ninv);  // -tbar / a.a
  const f2 y0 = fma2(s, G.a0, ub0), y1 = fma2(s, G.a1, ub1);
  const f2 su0 = mul2(s, G.u0), su1 = mul2(s, G.u1);
  const f2 p0 = fma2(G.t, y0, su0), p1 = fma2(G.t, y1, su1);  // z y + abar
  const f2 sg = fma2(nd, G.tau, s);
  S.v[0] = fma2(G.dx, p0, S.v[0]);
  S.v[1] = fma2(G.dy, p0, S.v[1]);
  S.v[2] = fma2(G.dy, p1, S.v[2]);
  S.v[3] = add2(S.v[3], y0);
  S.v[4] = add2(S.v[4], y1);
  S.v[5] = add2(S.v[5], sg);
  S.v[6] = add2(S.v[6], fma2(G.tau, y0, su0));
  S.v[7] = add2(S.v[7], fma2(G.tau, y1, su1));
  S.v[8] = fma2(G.tau, add2(sg, s), S.v[8]);
  S.v[9] = add2(S.v[9], nd);
  if (COLOR) {
    S.v[Acc::kCol + 0] = fma2(what, Cb0, S.v[Acc::kCol + 0]);
    S.v[Acc::kCol + 1] = fma2(what, Cb1, S.v[Acc::kCol + 1]);
    S.v[Acc::kCol + 2] = fma2(what, Cb2, S.v[Acc::kCol + 2]);
  }
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// A Gaussian's gradients from its summed accumulators, X B of the header first: M = X B'
// in the offsets' frame (c = S c', S = [[1/fx, 0, xe], [0, 1/fy, ye], [0, 0, 1]]), whose
// lower entries were accumulated.  Then X B = S M, Lbar = lower(R^T (X B) Q) with Q =
// B^-1 A from the prologue, mubar = R^-1 mbar, and the pose: Rbar = (X B) B^T R^-T -
// (R^-T mu) mubar^T (+ the normal's term), tbar = mbar, as functions of a general R (A =
// R L, m = R^-T mu + t).
// X itself, times A, would be the same, but its rounding is multiplied by the axis ratio
// there, while the columns of M along the short axes were summed directly.  The upper
// entry M01 still cancels for needles: flat Gaussians take it in float pairs.
// Discs, alpha's upstream alone, K = 24, against FP64 (world-frame form / X A / now):
// poses at ratio 100 2.4e-6 / 8.6e-5 / 1.5e-6, at 1000 3.6e-6 / 5.3e-3 / 3.4e-6; L at 1000 2.0e-6 /
// 5.4e-5 / 5.5e-7.  Orbit 650.8 -> 655 us, 9 views of 257x191 with colours 166 -> 168.6.
template <bool NORMALS, bool COLOR, bool POSE>
__device__ __forceinline__ void bwd_finalise(const Scene& s, const DevView& V, const float4* __restrict__ records,
                                             const float* view_inv, int g, const float* acc, bool want_pose, float gm[3],
                                             float gL[6], float& glam, float pose_g[12]) {
  using Acc = BwdAcc2<NORMALS, COLOR, POSE>;
  const long long gg = V.gauss_off + g;
  const float* rec = reinterpret_cast<const float*>(records) +
                     2 * kCamF2 * ((static_cast<long long>(V.rec_off) + g) >> 1) + (g & 1);
  const float pex = -rec[0], pey = -rec[2], B00 = rec[4], B10 = rec[6], e0 = rec[12], B11 = rec[14],
              e1 = rec[16], ee = rec[22], rho0 = rec[28], rho1 = rec[30];
  const float Y0 = acc[3], Y1 = acc[4], Kp = acc[8];
  // lower entries of X B' in the offsets' frame
  const float b00 = fmaf(-rho0, Y0, acc[0]), b10 = fmaf(-rho1, Y0, acc[1]), b11 = fmaf(-rho1, Y1, acc[2]);
  const float b20 = acc[6], b21 = acc[7];
  const float i0 = B00 != 0.f ? 1.0f / B00 : 0.f, i1 = B11 != 0.f ? 1.0f / B11 : 0.f;
  const float X22 = Kp;
  float X21, X20, M01;
  if ((__float_as_int(rec[26]) & kCamFlatter) == 0) {
    X21 = fmaf(-X22, e1, b21) * i1;
    const float X11 = fmaf(-X21, e1, b11) * i1;
    X20 = fmaf(-X22, e0, fmaf(-X21, B10, b20)) * i0;
    const float X10 = fmaf(-X21, e0, fmaf(-X11, B10, b10)) * i0;
    M01 = fmaf(X10, B11, X20 * e1);
  } else {
    const FF j0 = B00 != 0.f ? ff_rcp(FF{B00, 0.f}) : FF{0.f, 0.f}, j1 = B11 != 0.f ? ff_rcp(FF{B11, 0.f}) : FF{0.f, 0.f};
    const FF Y21 = (FF{b21, 0.f} - ff_prod(X22, e1)) * j1;
    const FF Y11 = (FF{b11, 0.f} - Y21 * e1) * j1;
    const FF Y20 = (FF{b20, 0.f} - ff_prod(X22, e0) - Y21 * B10) * j0;
    const FF Y10 = (FF{b10, 0.f} - Y11 * B10 - Y21 * e0) * j0;
    X21 = Y21.h;
    X20 = Y20.h;
    M01 = (Y10 * B11 + Y20 * e1).h;
  }
  const float e2 = sqrtf(ee);
  const float M[9] = {b00, M01, X20 * e2, b10, b11, X21 * e2, b20, b21, X22 * e2};
  const float ifx = 1.0f / V.fx, ify = 1.0f / V.fy, px = pex - V.cx, py = pey - V.cy;
  const float xe = px * ifx, ye = py * ify;
  float R[9], tp[3];
  load_pose(s.poses, V.pose, R, tp);
  const float4* qr = s.qrec + kCamQFloat4 * (static_cast<long long>(V.rec_off) + g);
  const float4 qa = qr[0], qb = qr[1], qc = qr[2];
  const float Q[9] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w, qc.x};
  float XA[9];  // (X B) Q
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float XB[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
      XB[c] = kCamScale * (a == 0 ? fmaf(ifx, M[c], xe * M[6 + c]) : a == 1 ? fmaf(ify, M[3 + c], ye * M[6 + c]) : M[6 + c]);
#pragma unroll
    for (int c = 0; c < 3; ++c) XA[3 * a + c] = fmaf(XB[2], Q[6 + c], fmaf(XB[1], Q[3 + c], XB[0] * Q[c]));
  }
  auto RtXA = [&](int a, int c) { return fmaf(R[6 + a], XA[6 + c], fmaf(R[3 + a], XA[3 + c], R[a] * XA[c])); };
  gL[0] = RtXA(0, 0);
  gL[1] = RtXA(1, 0);
  gL[2] = RtXA(1, 1);
  gL[3] = RtXA(2, 0);
  gL[4] = RtXA(2, 1);
  gL[5] = RtXA(2, 2);
  glam = -acc[9] / (kTwoLn2 * s.weights[gg]);
  // mbar = -B sum y; B's last row from e0, e1
  const float B20 = fmaf(-B10, py, fmaf(-B00, px, e0)), B21 = fmaf(-B11, py, e1);
  float mb[3];
  mb[0] = -V.fx * B00 * Y0;
  mb[1] = -V.fy * fmaf(B11, Y1, B10 * Y0);
  mb[2] = -fmaf(ee, acc[5], fmaf(B21, Y1, B20 * Y0));
#pragma unroll
  for (int c = 0; c < 3; ++c)
    gm[c] = fmaf(view_inv[3 * c + 2], mb[2], fmaf(view_inv[3 * c + 1], mb[1], view_inv[3 * c] * mb[0]));
  if (!POSE || !want_pose) return;
  const float mu0 = s.means[3 * gg], mu1 = s.means[3 * gg + 1], mu2 = s.means[3 * gg + 2];
  float T[9];
  if (NORMALS) {  // sum what (n . Nbar) n n^T, the third component from n . c = 0, its trace 0
    const float T00 = acc[Acc::kT], T01 = acc[Acc::kT + 1], T11 = acc[Acc::kT + 2];
    const float V0 = fmaf(px, T00, fmaf(py, T01, acc[Acc::kT + 3])), V1 = fmaf(px, T01, fmaf(py, T11, acc[Acc::kT + 4]));
    T[0] = V.fx * V.fx * T00;
    T[4] = V.fy * V.fy * T11;
    T[1] = T[3] = V.fx * V.fy * T01;
    T[2] = T[6] = -V.fx * V0;
    T[5] = T[7] = -V.fy * V1;
    T[8] = -(T[0] + T[4]);
  }
  // (X B) B^T in the camera frame: S (M B'^T) S^-1
  float W[9], G[9];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    W[3 * a] = M[3 * a] * B00;
    W[3 * a + 1] = fmaf(M[3 * a + 1], B11, M[3 * a] * B10);
    W[3 * a + 2] = fmaf(M[3 * a + 2], e2, fmaf(M[3 * a + 1], e1, M[3 * a] * e0));
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float u[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
      u[c] = a == 0 ? fmaf(ifx, W[c], xe * W[6 + c]) : a == 1 ? fmaf(ify, W[3 + c], ye * W[6 + c]) : W[6 + c];
    G[3 * a] = u[0] * V.fx;
    G[3 * a + 1] = u[1] * V.fy;
    G[3 * a + 2] = fmaf(-px, u[0], fmaf(-py, u[1], u[2]));
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // row a of R^-T mu
    const float rm = fmaf(view_inv[6 + a], mu2, fmaf(view_inv[3 + a], mu1, view_inv[a] * mu0));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float x = fmaf(-rm, gm[c], fmaf(G[3 * a + 2], view_inv[3 * c + 2],
                                      fmaf(G[3 * a + 1], view_inv[3 * c + 1], G[3 * a] * view_inv[3 * c])));
      if (NORMALS) x += fmaf(T[3 * a + 2], R[6 + c], fmaf(T[3 * a + 1], R[3 + c], T[3 * a] * R[c]));
      pose_g[3 * a + c] += x;
    }
    pose_g[9 + a] += mb[a];
  }
}

// CL = 2: launched as clusters of two CTAs, the two Gaussian blocks of one ray tile
// (grid mode, every view of the batch in two blocks); CL = 1: no cluster.
template <bool NORMALS, int NFLOW, bool COLOR = false, bool POSE = true, int CL = 1, class B = Batch>
__global__ void __launch_bounds__(kBwdMaxThreads, kBwdMinBlocks)
    backward_kernel(const __grid_constant__ B batch, Scene s, Consts k, const float4* __restrict__ records,
                    BwdIn in, BwdOut out, int ray_tile, int* counter) {
  pdl_enter();
  extern __shared__ float4 bsm[];
  constexpr int NPV = 12 * (1 + NFLOW);  // pose values reduced per CTA
  __shared__ float pose_ray[kBwdMaxThreads / 32][NPV];  // per-warp sums of the per-ray pose terms
  __shared__ float pose_gau[kBwdMaxThreads / 32][12];   // per-warp sums of the per-Gaussian pose terms
  __shared__ float view_inv[9];                         // R^-1 of the view's pose
  __shared__ int s_item;
  if (CL == 2) cluster_arrive();  // this CTA runs: its shared memory may be written by its peer

  for (int round = 0;; ++round) {
  const int item = next_item(counter, round, &s_item);
  if (item < 0 || item >= batch.n_items) break;
  int local;
  const int vi = find_item(batch, item, local);
  const DevView& V = batch.v[vi];
  const int tile = local / V.n_gblocks;
  const int gb = local - tile * V.n_gblocks;
  const int P = V.P;
  const int rt = V.rt > 0 ? V.rt : ray_tile;  // the view's tiles are balanced: rt <= ray_tile
  const int pix0 = tile * rt;
  const int nr = min(rt, P - pix0);
  const int tid = threadIdx.x;
  const int T = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5;
  const long long off = V.pix_off;
  const bool want_pose = out.gposes != nullptr;
  // In a cluster (CL = 2) each CTA builds the records of its half of the tile's
  // rays and writes them to both CTAs (its own shared memory and, through
  // distributed shared memory, its peer's), so a ray's record is built once, not
  // once per Gaussian block.
  const int crank = CL == 2 ? static_cast<int>(cluster_ctarank()) : 0;
  const int r_lo = CL == 2 ? (nr * crank) / 2 : 0;
  const int r_hi = CL == 2 ? (nr * (crank + 1)) / 2 : nr;
  // per-ray pose terms: once per ray (by the CTA that builds its record)
  const bool ray_pose = want_pose && (CL == 2 || gb == 0);

  // ---------------- phase 1: per-ray records (and the per-ray pose terms)
  {
    float R[9], tp[3];
    load_pose(s.poses, V.pose, R, tp);
    const float o0 = -fmaf(R[6], tp[2], fmaf(R[3], tp[1], R[0] * tp[0]));
    const float o1 = -fmaf(R[7], tp[2], fmaf(R[4], tp[1], R[1] * tp[0]));
    const float o2 = -fmaf(R[8], tp[2], fmaf(R[5], tp[1], R[2] * tp[0]));
    if (tid < 9) {  // entry (a, b) of R^-1 = cof(R)^T / det(R)
      const int a = tid / 3, b = tid % 3;
      auto at = [&](int i, int j) { return __ldg(s.poses + 12 * static_cast<long long>(V.pose) + 3 * (i % 3) + j % 3); };
      const float cof = fmaf(at(b + 1, a + 1), at(b + 2, a + 2), -(at(b + 1, a + 2) * at(b + 2, a + 1)));
      const float det = fmaf(R[0], fmaf(R[4], R[8], -(R[5] * R[7])),
                             fmaf(R[1], fmaf(R[5], R[6], -(R[3] * R[8])), R[2] * fmaf(R[3], R[7], -(R[4] * R[6]))));
      view_inv[tid] = cof / det;
    }
    float pose_acc[NPV];
#pragma unroll
    for (int i = 0; i < NPV; ++i) pose_acc[i] = 0.f;
    float Rj[NFLOW > 0 ? NFLOW : 1][9], tj[NFLOW > 0 ? NFLOW : 1][3];
    bool has_t[NFLOW > 0 ? NFLOW : 1];
#pragma unroll
    for (int j = 0; j < NFLOW; ++j) {
      const int tg = j == 0 ? V.tgt0 : V.tgt1;
      has_t[j] = tg >= 0 && in.g_flow != nullptr;
      if (has_t[j]) load_pose(s.poses, tg, Rj[j], tj[j]);
    }
    if (CL == 2) cluster_wait();  // the peer runs: its shared memory may be written (clusters take one item)
    for (int r = r_lo + tid; r < r_hi; r += T) {
      const int p = pix0 + r;
      const CamRay ray = cam_ray(V, ray_pixel(V, p));
      const float vc[3] = {ray.x * ray.ilen, ray.y * ray.ilen, ray.ilen};
      float v[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) v[c] = fmaf(R[6 + c], vc[2], fmaf(R[3 + c], vc[1], R[c] * vc[0]));
      const float D = in.depth[off + p];
      const float* sv = in.saved + 3 * off;
      const float lse2 = sv[p];
      const float Sd = sv[P + p];
      const float gD = in.g_depth ? in.g_depth[off + p] : 0.f;
      const float gA = in.g_alpha ? in.g_alpha[off + p] : 0.f;
      float pb0 = 0.f, pb1 = 0.f, pb2 = 0.f;
      if (NFLOW > 0) {
        const float p0 = fmaf(v[0], D, o0), p1 = fmaf(v[1], D, o1), p2 = fmaf(v[2], D, o2);
        const float* gf = in.g_flow + 2 * NFLOW * off;
#pragma unroll
        for (int j = 0; j < NFLOW; ++j) {
          if (!has_t[j]) continue;
          const float X0 = fmaf(Rj[j][2], p2, fmaf(Rj[j][1], p1, fmaf(Rj[j][0], p0, tj[j][0])));
          const float X1 = fmaf(Rj[j][5], p2, fmaf(Rj[j][4], p1, fmaf(Rj[j][3], p0, tj[j][1])));
          const float X2 = fmaf(Rj[j][8], p2, fmaf(Rj[j][7], p1, fmaf(Rj[j][6], p0, tj[j][2])));
          const float iz = 1.0f / X2;
          const float gu = gf[(2 * j) * P + p], gv = gf[(2 * j + 1) * P + p];
          const float Xb0 = gu * V.fx * iz;
          const float Xb1 = gv * V.fy * iz;
          const float Xb2 = -(Xb0 * X0 + Xb1 * X1) * iz;
          pb0 += fmaf(Rj[j][6], Xb2, fmaf(Rj[j][3], Xb1, Rj[j][0] * Xb0));
          pb1 += fmaf(Rj[j][7], Xb2, fmaf(Rj[j][4], Xb1, Rj[j][1] * Xb0));
          pb2 += fmaf(Rj[j][8], Xb2, fmaf(Rj[j][5], Xb1, Rj[j][2] * Xb0));
          if (ray_pose) {
            float* pa = pose_acc + 12 * (1 + j);
            const float Xb[3] = {Xb0, Xb1, Xb2};
            const float pp[3] = {p0, p1, p2};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
#pragma unroll
              for (int c = 0; c < 3; ++c) pa[3 * a + c] = fmaf(Xb[a], pp[c], pa[3 * a + c]);
              pa[9 + a] += Xb[a];
            }
          }
        }
      }
      const float Dbar = fmaf(v[2], pb2, fmaf(v[1], pb1, fmaf(v[0], pb0, gD)));
      if (ray_pose && NFLOW > 0) {
        // p = o + v D with o = -R^T t, v = R^T vc:  Rbar += (D vc - t) pbar^T, tbar -= R pbar
        const float w[3] = {fmaf(D, vc[0], -tp[0]), fmaf(D, vc[1], -tp[1]), fmaf(D, vc[2], -tp[2])};
        const float pb[3] = {pb0, pb1, pb2};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
#pragma unroll
          for (int c = 0; c < 3; ++c) pose_acc[3 * a + c] = fmaf(w[a], pb[c], pose_acc[3 * a + c]);
          pose_acc[9 + a] -= fmaf(R[3 * a + 2], pb2, fmaf(R[3 * a + 1], pb1, R[3 * a] * pb0));
        }
      }
      float Nb0 = 0.f, Nb1 = 0.f, Nb2 = 0.f;
      if (NORMALS && in.g_normal != nullptr) {
        const float* nr3 = in.normal + 3 * off;
        const float* gn3 = in.g_normal + 3 * off;
        const float nc[3] = {nr3[p], nr3[P + p], nr3[2 * P + p]};
        const float gn[3] = {gn3[p], gn3[P + p], gn3[2 * P + p]};
        const float Nn = sv[2 * P + p];
        // Camera frame throughout: Nbar = (gn - (gn . n) n) / |N|.  The rendered normal is
        // R n_f with n_f formed in the world frame, so a change of R that is not a
        // rotation also acts through R^-1 g: with the pair terms of phase 2 that adds
        // [(gn . n) n n^T + sum what (n_i . Nbar) n_i n_i^T] R to the pose's gradient.
        const float sdot = fmaf(nc[2], gn[2], fmaf(nc[1], gn[1], nc[0] * gn[0]));
        if (ray_pose) {
          float nR[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) nR[c] = sdot * fmaf(R[6 + c], nc[2], fmaf(R[3 + c], nc[1], R[c] * nc[0]));
#pragma unroll
          for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int c = 0; c < 3; ++c) pose_acc[3 * a + c] = fmaf(nc[a], nR[c], pose_acc[3 * a + c]);
        }
        if (Nn > 0.f) {
          const float iN = 1.0f / Nn;
          Nb0 = fmaf(-sdot, nc[0], gn[0]) * iN;
          Nb1 = fmaf(-sdot, nc[1], gn[1]) * iN;
          Nb2 = fmaf(-sdot, nc[2], gn[2]) * iN;
        }
      }
      // Nbar is orthogonal to N, so the softmax centring terms are Dbar D and, in colour
      // mode, Cbar . C (the blended colour's).
      float Cb[3] = {0.f, 0.f, 0.f}, CC = 0.f;
      if (COLOR && in.g_color != nullptr) {
        const float* gc3 = in.g_color + 3 * off;
        const float* cp3 = in.color + 3 * off;
#pragma unroll
        for (int k3 = 0; k3 < 3; ++k3) {
          Cb[k3] = gc3[k3 * P + p];
          CC = fmaf(Cb[k3], cp3[k3 * P + p], CC);
        }
      }
      const float KA = kTwoLn2 * gA * expf(-Sd);
      const float Dq = __fmul_rn(D, ray.ilen);  // D / |c|, corrected by its remainder
      const float Dz = Dbar * ray.len, nD = -__fmaf_rn(__fmaf_rn(-Dq, ray.len, D), ray.ilen, Dq);
      constexpr int NR = ray_rec2<NORMALS, COLOR>();
      const float K2 = __fmul_rn(k.K2, ray.len), b2 = k.b2e * ray.len;
      float4 rec[NR];
      rec[0] = make_float4(ray.px, ray.px, ray.py, ray.py);
      rec[1] = make_float4(-lse2, -lse2, K2, K2);
      rec[2] = make_float4(Dz, Dz, nD, nD);
      rec[3] = make_float4(-KA, -KA, -b2, -b2);
      if constexpr (NORMALS) {
        const float n0 = V.fx * fmaf(-ray.x, Nb2, Nb0), n1 = V.fy * fmaf(-ray.y, Nb2, Nb1);
        const float m00 = -V.fx * V.fx * fmaf(ray.x, ray.x, 1.0f), m01 = -V.fx * V.fy * (ray.x * ray.y);
        const float m11 = -V.fy * V.fy * fmaf(ray.y, ray.y, 1.0f);
        rec[4] = make_float4(n0, n0, n1, n1);
        rec[5] = make_float4(m00, m00, m01, m01);
        rec[6] = make_float4(m11, m11, 0.f, 0.f);
      }
      if constexpr (COLOR) {
        rec[NR - 2] = make_float4(Cb[0], Cb[0], Cb[1], Cb[1]);
        rec[NR - 1] = make_float4(Cb[2], Cb[2], -CC, -CC);
      }
      float4* rr = bsm + NR * r;
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        rr[i] = rec[i];
        if (CL == 2) st_cluster_f4(rr + i, crank ^ 1, rec[i]);
      }
    }
    // Reduce the per-ray pose terms now, so that they hold no registers in the loop.
    if (want_pose) {
#pragma unroll
      for (int i = 0; i < NPV; ++i) {
        const float x = warp_sum(pose_acc[i]);
        if (lane == 0) pose_ray[warp][i] = x;
      }
    }
  }
  // the records (the cluster's, through distributed shared memory) are complete
  if (CL == 2)
    cluster_sync();
  else
    __syncthreads();

  // ---------------- phase 2: Gaussian-parallel pair loop (two Gaussians per thread)
  const int GB = V.GB, S = V.S;
  const int GB2 = (GB + 1) / 2;  // threads per ray subgroup
  const int gl2 = tid % GB2;
  const int sg = tid / GB2;
  const int g0 = gb * GB + 2 * gl2;  // lane 0 Gaussian (GB is even unless there is one block: whole records)
  const bool active = (sg < S) && (g0 < V.K);
  using Acc = BwdAcc2<NORMALS, COLOR, POSE>;
  Acc A;
#pragma unroll
  for (int i = 0; i < Acc::kN; ++i) A.v[i] = dup(0.f);
  const long long rec0 = static_cast<long long>(V.rec_off) + (active ? g0 : 0);
  const CamRec2 gr = cam_load(reinterpret_cast<const ulonglong2*>(records + kRecFloat4 * rec0));
  constexpr unsigned long long kFlat = (static_cast<unsigned long long>(kCamFlatter) << 32) | kCamFlatter;
  const bool flat = NORMALS && __any_sync(0xffffffffu, active && (gr.flags & kFlat) != 0);
  if (active) {
    const f2 nB1 = dup(-k.beta1), nB1s = dup(-kTwoLn2 * k.beta1), tiny = dup(-1e-30f);
    const ulonglong2* rays = reinterpret_cast<const ulonglong2*>(bsm);
    constexpr int NR = ray_rec2<NORMALS, COLOR>(), kUnroll = bwd_unroll<NORMALS>();
    f2 c0 = dup(0.f), c1 = c0, c2 = c0;  // the two Gaussians' colours, one per lane
    if (COLOR) {
      const ulonglong2* cr = reinterpret_cast<const ulonglong2*>(s.crec + rec0);
      c0 = as_f2(cr[0].x);
      c1 = as_f2(cr[0].y);
      c2 = as_f2(cr[1].x);
    }
    // with colours one loop serves both: two spilled 180 bytes per thread (54 views of
    // 1025x675 at K = 79 13.50 against 12.34 ms; without colours one loop is 1 to 3 % slower)
    if (COLOR || !flat) {
#pragma unroll kUnroll
      for (int r = sg; r < nr; r += S)
        bwd_pair2<NORMALS, COLOR, POSE, false>(A, gr, rays + NR * r, nB1, nB1s, tiny, c0, c1, c2, flat);
    } else if (NORMALS) {
#pragma unroll 1
      for (int r = sg; r < nr; r += S)
        bwd_pair2<NORMALS, COLOR, POSE, NORMALS>(A, gr, rays + NR * r, nB1, nB1s, tiny, c0, c1, c2);
    }
  }
  __syncthreads();  // ray records are dead; the shared memory is reused below

  // ---------------- phase 3: combine ray subgroups, finalise per Gaussian
  constexpr int NV = Acc::kN;          // sums per Gaussian
  constexpr int NC = COLOR ? 13 : 10;  // gradient values per Gaussian in a partial slot
  f2* red = reinterpret_cast<f2*>(bsm);  // [sum][thread]
  if (sg < S) {
#pragma unroll
    for (int i = 0; i < NV; ++i) red[i * T + tid] = A.v[i];
  }
  __syncthreads();
  float* slot = nullptr;
  if (out.partials) {
    const int t = out.slots > 0 ? tile % out.slots : tile;
    slot = out.partials + V.part_off + static_cast<long long>(t * V.n_gblocks + gb) * V.slot_floats;
  }
  const bool accumulate = out.slots > 0;
  float pose_g[12];
#pragma unroll
  for (int i = 0; i < 12; ++i) pose_g[i] = 0.f;
  for (int gi = tid; gi < GB; gi += T) {  // one Gaussian per thread
    const int g = gb * GB + gi;
    float gm[3] = {0, 0, 0}, gL[6] = {0, 0, 0, 0, 0, 0}, glam = 0.f, gcol[3] = {0, 0, 0};
    if (g < V.K) {
      float acc[NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) acc[i] = 0.f;
      for (int s2 = 0; s2 < S; ++s2) {
        const float* d = reinterpret_cast<const float*>(red + s2 * GB2 + (gi >> 1)) + (gi & 1);
#pragma unroll
        for (int i = 0; i < NV; ++i) acc[i] += d[2 * i * T];
      }
      bwd_finalise<NORMALS, COLOR, POSE>(s, V, records, view_inv, g, acc, want_pose, gm, gL, glam, pose_g);
      if (COLOR) {
#pragma unroll
        for (int k3 = 0; k3 < 3; ++k3) gcol[k3] = acc[Acc::kCol + k3];
      }
    }
    if (slot == nullptr) {
      if (g < V.K) {
        const long long gg = V.gauss_off + g;
        atomicAdd(out.gmeans + 3 * gg + 0, gm[0]);
        atomicAdd(out.gmeans + 3 * gg + 1, gm[1]);
        atomicAdd(out.gmeans + 3 * gg + 2, gm[2]);
#pragma unroll
        for (int i = 0; i < 6; ++i) atomicAdd(out.gchol + 6 * gg + i, gL[i]);
        atomicAdd(out.gweights + gg, glam);
        if (COLOR) {
#pragma unroll
          for (int k3 = 0; k3 < 3; ++k3) atomicAdd(out.gcolors + 3 * gg + k3, gcol[k3]);
        }
      }
    } else {
      float* d = slot + NC * gi;
      const float v[13] = {gm[0], gm[1], gm[2], gL[0], gL[1], gL[2], gL[3], gL[4], gL[5], glam, gcol[0], gcol[1], gcol[2]};
      if (!accumulate) {
#pragma unroll
        for (int i = 0; i < NC; ++i) d[i] = v[i];
      } else if (g < V.K) {
#pragma unroll
        for (int i = 0; i < NC; ++i) atomicAdd(d + i, v[i]);
      }
    }
  }

  // ---------------- phase 4: pose gradient of this CTA
  if (want_pose) {
#pragma unroll
    for (int i = 0; i < 12; ++i) {
      const float x = warp_sum(pose_g[i]);
      if (lane == 0) pose_gau[warp][i] = x;
    }
    __syncthreads();
    if (tid < NPV) {
      float x = 0.f;
      const int nw = (T + 31) / 32;
      for (int w = 0; w < nw; ++w) x += pose_ray[w][tid] + (tid < 12 ? pose_gau[w][tid] : 0.f);
      if (slot != nullptr && accumulate) {
        atomicAdd(slot + NC * GB + tid, x);
      } else if (slot != nullptr) {
        slot[NC * GB + tid] = x;
      } else {
        const int j = tid / 12 - 1;
        const int pidx = j < 0 ? V.pose : (j == 0 ? V.tgt0 : V.tgt1);
        if (pidx >= 0) atomicAdd(out.gposes + 12 * static_cast<long long>(pidx) + tid % 12, x);
      }
    }
  }
  }  // item loop
}

template <bool NORMALS, bool COLOR, bool POSE>
static int bwd_smem_bytes(int ray_tile, int threads) {
  return std::max(ray_tile * ray_rec2<NORMALS, COLOR>() * static_cast<int>(sizeof(float4)),
                  threads * acc_count<NORMALS, COLOR, POSE>() * static_cast<int>(sizeof(f2)));
}

template <bool NORMALS, int NFLOW, bool COLOR = false, bool POSE = true, int CL = 1, class B = Batch>
static cudaError_t prepare_bwd_t(int smem) {
  // Dynamic plus static shared memory above the 48 KB default needs the opt-in; the static
  // part is about 1 KB.
  if (smem > 46 * 1024)
    return cudaFuncSetAttribute(backward_kernel<NORMALS, NFLOW, COLOR, POSE, CL, B>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return cudaSuccess;
}

template <bool NORMALS, int NFLOW>
static int bwd_ctas_per_sm_t(int ray_tile, int threads) {
  const int smem = bwd_smem_bytes<NORMALS, false, true>(ray_tile, threads);
  if (prepare_bwd_t<NORMALS, NFLOW>(smem) != cudaSuccess) return 1;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, backward_kernel<NORMALS, NFLOW>, threads, smem) !=
      cudaSuccess)
    return 1;
  return n > 0 ? n : 1;
}

// Cluster size of a grid-mode backward launch: 2 when every view of the batch runs
// as two Gaussian blocks (then each tile's two items are consecutive and 2-aligned,
// one cluster), else 1 (no cluster).
template <class B>
static int bwd_cluster_size(const B& b) {
  int C = 0;
  for (int i = 0; i < b.n_views; ++i) {
    const DevView& v = b.v[i];
    if (v.n_tiles <= 0) continue;
    if (C == 0) C = v.n_gblocks;
    if (v.n_gblocks != C) return 1;
  }
  if (C != 2 || b.n_items % C != 0) return 1;
  for (int j = 0; j < b.n_views; ++j)
    if (b.order_begin[j] % C != 0) return 1;
  return C;
}

template <bool NORMALS, int NFLOW, bool COLOR = false, bool POSE = true, class B>
static cudaError_t launch_bwd_s(const B& b, const Scene& s, const Consts& c, const float4* records,
                                int ray_tile, int threads, const BwdIn& in, const BwdOut& out, int* counter,
                                cudaStream_t st) {
  const int smem = bwd_smem_bytes<NORMALS, COLOR, POSE>(ray_tile, threads);
  cudaError_t e = prepare_bwd_t<NORMALS, NFLOW, COLOR, POSE, 1, B>(smem);
  if (e != cudaSuccess) return e;
  int grid = b.n_items;
  if (counter) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    grid = std::min(b.n_items, std::max(1, sms) * bwd_ctas_per_sm_t<NORMALS, NFLOW>(ray_tile, threads));
  }
  if constexpr (!COLOR) {
    if (counter == nullptr && bwd_cluster_size(b) == 2) {
      e = prepare_bwd_t<NORMALS, NFLOW, COLOR, POSE, 2, B>(smem);
      if (e != cudaSuccess) return e;
      return launch_kernel(backward_kernel<NORMALS, NFLOW, COLOR, POSE, 2, B>, dim3(grid), dim3(threads), smem,
                           st, 2, b, s, c, records, in, out, ray_tile, counter);
    }
  }
  return launch_kernel(backward_kernel<NORMALS, NFLOW, COLOR, POSE, 1, B>, dim3(grid), dim3(threads), smem, st,
                       1, b, s, c, records, in, out, ray_tile, counter);
}

template <bool NORMALS, int NFLOW, class B>
static cudaError_t launch_bwd_t(const B& b, const Scene& s, const Consts& c, const float4* records,
                                int ray_tile, int threads, const BwdIn& in, const BwdOut& out, int* counter,
                                cudaStream_t st) {
  if (out.gcolors != nullptr)
    return launch_bwd_s<NORMALS, NFLOW, true>(b, s, c, records, ray_tile, threads, in, out, counter, st);
  if (out.gposes == nullptr)
    return launch_bwd_s<NORMALS, NFLOW, false, false>(b, s, c, records, ray_tile, threads, in, out, counter,
                                                              st);
  return launch_bwd_s<NORMALS, NFLOW>(b, s, c, records, ray_tile, threads, in, out, counter, st);
}

template <class B>
static cudaError_t launch_backward_t(const B& b, const Scene& s, const Consts& c, const float4* records,
                                     bool normals, int n_flow, int ray_tile, int threads, const BwdIn& in,
                                     const BwdOut& out, int* counter, cudaStream_t st) {
  if (normals) {
    if (n_flow == 0) return launch_bwd_t<true, 0>(b, s, c, records, ray_tile, threads, in, out, counter, st);
    if (n_flow == 1) return launch_bwd_t<true, 1>(b, s, c, records, ray_tile, threads, in, out, counter, st);
    return launch_bwd_t<true, 2>(b, s, c, records, ray_tile, threads, in, out, counter, st);
  }
  if (n_flow == 0) return launch_bwd_t<false, 0>(b, s, c, records, ray_tile, threads, in, out, counter, st);
  if (n_flow == 1) return launch_bwd_t<false, 1>(b, s, c, records, ray_tile, threads, in, out, counter, st);
  return launch_bwd_t<false, 2>(b, s, c, records, ray_tile, threads, in, out, counter, st);
}
cudaError_t launch_backward(const Batch& b, const Scene& s, const Consts& c, const float4* records, bool normals,
                            int n_flow, int ray_tile, int threads, const BwdIn& in, const BwdOut& out,
                            int* counter, cudaStream_t st) {
  return launch_backward_t(b, s, c, records, normals, n_flow, ray_tile, threads, in, out, counter, st);
}
cudaError_t launch_backward(const BigBatch& b, const Scene& s, const Consts& c, const float4* records, bool normals,
                            int n_flow, int ray_tile, int threads, const BwdIn& in, const BwdOut& out,
                            int* counter, cudaStream_t st) {
  return launch_backward_t(b, s, c, records, normals, n_flow, ray_tile, threads, in, out, counter, st);
}

int backward_ctas_per_sm(bool normals, int n_flow, int ray_tile, int threads) {
  (void)normals;
  (void)n_flow;
  return bwd_ctas_per_sm_t<true, 1>(ray_tile, threads);
}

// ------------------------------------------------- zeroing of the outputs
// One launch clears the status word and every gradient output before the
// backward kernels accumulate into them.
__global__ void zero_kernel(ZeroJob job) {
  pdl_enter();
  const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
  long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  for (int b = 0; b < ZeroJob::kMax; ++b) {
    if (job.ptr[b] == nullptr) continue;
    for (long long j = i; j < job.n[b]; j += stride) job.ptr[b][j] = 0.f;
  }
}

cudaError_t launch_zero(const ZeroJob& job, cudaStream_t st) {
  return launch_kernel(zero_kernel, dim3(2 * 152), dim3(256), 0, st, 1, job);
}

// ------------------------------------------- deterministic second stage
// One warp per output value: lane l adds slots l, l+32, l+64, ... in order, then a
// fixed butterfly combines the lanes, so the result does not depend on timing.
__device__ __forceinline__ float warp_sum_fixed(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Gaussian gradients: warp w handles (Gaussian g, component comp), w = g * nc + comp
// (nc = 10, or 13 with colours: means 3, chol 6, weight 1, colour 3).
__device__ __forceinline__ float* gauss_grad(const BwdOut& out, long long g, int comp) {
  if (comp < 3) return out.gmeans + 3 * g + comp;
  if (comp < 9) return out.gchol + 6 * g + comp - 3;
  if (comp == 9) return out.gweights + g;
  return out.gcolors + 3 * g + comp - 10;
}

template <class B>
__global__ void reduce_gauss_kernel(const __grid_constant__ B batch, BwdOut out, long long n_gauss, int nc) {
  pdl_enter();
  const long long w = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= n_gauss * nc) return;  // whole warps exit together
  const long long g = w / nc;
  const int comp = static_cast<int>(w - g * nc);
  float acc = 0.f;
  bool hit = false;
  for (int v = 0; v < batch.n_views; ++v) {
    const DevView& V = batch.v[v];
    if (g < V.gauss_off || g >= V.gauss_off + V.K) continue;
    hit = true;
    const int gi = static_cast<int>(g - V.gauss_off);
    const int gbk = gi / V.GB, gl = gi - gbk * V.GB;
    for (int t = lane; t < V.n_tiles; t += 32)
      acc += out.partials[V.part_off + static_cast<long long>(t * V.n_gblocks + gbk) * V.slot_floats + nc * gl + comp];
  }
  acc = warp_sum_fixed(acc);
  if (hit && lane == 0) *gauss_grad(out, g, comp) += acc;
}

// Pose gradients: warp w handles (pose p, component comp), w = p * 12 + comp.
template <class B>
__global__ void reduce_pose_kernel(const __grid_constant__ B batch, BwdOut out, int n_poses, int n_flow, int nc) {
  pdl_enter();
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= n_poses * 12) return;
  const int p = w / 12, comp = w % 12;
  float acc = 0.f;
  for (int v = 0; v < batch.n_views; ++v) {
    const DevView& V = batch.v[v];
    for (int j = -1; j < n_flow; ++j) {
      const int pidx = j < 0 ? V.pose : (j == 0 ? V.tgt0 : V.tgt1);
      if (pidx != p) continue;
      const int part = 12 * (j + 1) + comp;
      const int nslots = V.n_tiles * V.n_gblocks;
      for (int sl = lane; sl < nslots; sl += 32)
        acc += out.partials[V.part_off + static_cast<long long>(sl) * V.slot_floats + nc * V.GB + part];
    }
  }
  acc = warp_sum_fixed(acc);
  if (lane == 0) out.gposes[12 * static_cast<long long>(p) + comp] += acc;
}

// The slots of atomic mode, view by view: a thread adds the (at most kAccSlots) slots of
// one value of one view and adds that to the gradient, so the work follows what was
// rendered.  (A warp per value that looks for it in every view, as above, took 57 ms
// after 2.0 ms of adjoint for 256 objects of 1024 Gaussians, one 64x64 view each.)
template <class B>
__global__ void __launch_bounds__(256) add_slots_gauss_kernel(const __grid_constant__ B batch, BwdOut out, int nc) {
  pdl_enter();
  const DevView& V = batch.v[blockIdx.y];
  const long long e = blockIdx.x * 256ll + threadIdx.x;
  if (e >= static_cast<long long>(V.K) * nc) return;
  const int gi = static_cast<int>(e / nc), comp = static_cast<int>(e - static_cast<long long>(gi) * nc);
  const int gbk = gi / V.GB;
  const float* src = out.partials + V.part_off + static_cast<long long>(gbk) * V.slot_floats + nc * (gi - gbk * V.GB) + comp;
  const long long step = static_cast<long long>(V.n_gblocks) * V.slot_floats;
  const int n = min(out.slots, V.n_tiles);
  float acc = 0.f;
  for (int t = 0; t < n; ++t) acc += src[t * step];
  atomicAdd(gauss_grad(out, V.gauss_off + gi, comp), acc);
}
// A warp per value of a view's pose sums.
template <class B>
__global__ void __launch_bounds__(384) add_slots_pose_kernel(const __grid_constant__ B batch, BwdOut out, int n_flow, int nc) {
  pdl_enter();
  const DevView& V = batch.v[blockIdx.x];
  const int lane = threadIdx.x & 31, comp = threadIdx.x >> 5;
  const int nslots = min(out.slots, V.n_tiles) * V.n_gblocks;
  for (int j = -1; j < n_flow; ++j) {
    const int pidx = j < 0 ? V.pose : (j == 0 ? V.tgt0 : V.tgt1);
    if (pidx < 0) continue;
    const float* src = out.partials + V.part_off + nc * V.GB + 12 * (j + 1) + comp;
    float acc = 0.f;
    for (int sl = lane; sl < nslots; sl += 32) acc += src[static_cast<long long>(sl) * V.slot_floats];
    acc = warp_sum_fixed(acc);
    if (lane == 0) atomicAdd(out.gposes + 12 * static_cast<long long>(pidx) + comp, acc);
  }
}

template <class B>
static cudaError_t launch_backward_reduce_t(const B& b, int n_flow, long long n_gauss, int n_poses,
                                            const BwdOut& out, cudaStream_t st) {
  const int nc = out.gcolors != nullptr ? 13 : 10;
  if (out.slots > 0) {
    long long values = 0;
    for (int i = 0; i < b.n_views; ++i) values = std::max(values, static_cast<long long>(b.v[i].K) * nc);
    const dim3 grid(static_cast<unsigned>((values + 255) / 256), static_cast<unsigned>(b.n_views));
    const cudaError_t e = launch_kernel(add_slots_gauss_kernel<B>, grid, dim3(256), 0, st, 1, b, out, nc);
    if (e != cudaSuccess || out.gposes == nullptr) return e;
    return launch_kernel(add_slots_pose_kernel<B>, dim3(b.n_views), dim3(384), 0, st, 1, b, out, n_flow, nc);
  }
  const long long warps = n_gauss * nc;
  const dim3 grid(static_cast<unsigned>((warps * 32 + 255) / 256));
  const cudaError_t e = launch_kernel(reduce_gauss_kernel<B>, grid, dim3(256), 0, st, 1, b, out, n_gauss, nc);
  if (e != cudaSuccess || out.gposes == nullptr) return e;
  return launch_kernel(reduce_pose_kernel<B>, dim3((n_poses * 12 * 32 + 255) / 256), dim3(256), 0, st, 1, b, out,
                       n_poses, n_flow, nc);
}
cudaError_t launch_backward_reduce(const Batch& b, int n_flow, long long n_gauss, int n_poses, const BwdOut& out,
                                   cudaStream_t st) {
  return launch_backward_reduce_t(b, n_flow, n_gauss, n_poses, out, st);
}
cudaError_t launch_backward_reduce(const BigBatch& b, int n_flow, long long n_gauss, int n_poses, const BwdOut& out,
                                   cudaStream_t st) {
  return launch_backward_reduce_t(b, n_flow, n_gauss, n_poses, out, st);
}

}  // namespace fmb
