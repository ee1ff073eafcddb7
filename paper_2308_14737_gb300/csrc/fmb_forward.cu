// fmb_forward.cu -- prologue (per view x Gaussian records) and forward render
// kernel of the two-parameter Fuzzy Metaballs renderer.
//
// Formulation (paper Eq. 2, 3, 4, 7, 8, 17; Sec. 5 flow): the max-likelihood depth t
// along the ray, the Mahalanobis term q there, d = -q/2 + ln(lambda), delta = e^d, the
// weight exponent of Eq. 7 e = beta1 d - (beta2/eta) t, and the local normal
// Sigma^-1 (o + v t - mu) of Eq. 17, all in the camera-plane form of fmb_cam.cuh and
// in the log2 domain, so that the exponentials are single ex2 instructions.
#include <algorithm>

#include "fmb_cam.cuh"
#include "fmb_f32x2.cuh"
#include "fmb_internal.cuh"

namespace fmb {

constexpr int kFwdThreads = 128;
constexpr int kChunk = 256;  // Gaussians per shared-memory stage (16 KB)
// Minus the shift before a lane's first Gaussian.  Finite: the exponent of a Gaussian of
// weight 0 is -inf, which must leave its weight at 0 (not inf - inf).
constexpr float kNoShift = 3e38f;

// ------------------------------------------------------------------ prologue
// The world-frame kernels' records (fmb_world_*.cu, alpha compositing, point export,
// attribution).  One thread per (view, Gaussian): the record of unpack_rec.  The camera centre
// o = -R^T t and m = mu - o are formed as exact float pairs (error-free
// transformations), so that the per-pair residual can be evaluated to full fp32
// accuracy relative to its own size.  The same launch clears the arrays of `zero`
// (the backward's gradient outputs and status word, which its kernels then
// accumulate into), grid-stride over all its threads.
// The rest of a world-frame record from L and mu - o = mh + ml.
__device__ __forceinline__ void world_record(GaussRec& q, const float ml[3], float weight) {
  const float* L = q.L;
  q.b[0] = fmaf(L[3], q.mh[2], fmaf(L[1], q.mh[1], L[0] * q.mh[0]));
  q.b[1] = fmaf(L[4], q.mh[2], L[2] * q.mh[1]);
  q.b[2] = L[5] * q.mh[2];
  q.nbl[0] = -fmaf(L[3], ml[2], fmaf(L[1], ml[1], L[0] * ml[0]));
  q.nbl[1] = -fmaf(L[4], ml[2], L[2] * ml[1]);
  q.nbl[2] = -(L[5] * ml[2]);
  q.l2 = log2f(weight);
}

__device__ __forceinline__ void prologue_clear(int* status_to_clear, int* counter_to_clear, const ZeroJob& zero) {
  const long long stride = static_cast<long long>(gridDim.x) * gridDim.y * blockDim.x;
  const long long j0 = (static_cast<long long>(blockIdx.y) * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x;
  if (j0 == 0) {
    if (status_to_clear != nullptr) *status_to_clear = kDevOk;
    if (counter_to_clear != nullptr) *counter_to_clear = 0;
  }
  for (int b = 0; b < ZeroJob::kMax; ++b) {
    if (zero.ptr[b] == nullptr) continue;
    for (long long j = j0; j < zero.n[b]; j += stride) zero.ptr[b][j] = 0.f;
  }
}

template <class B>
__global__ void __launch_bounds__(128) prologue_kernel(const __grid_constant__ B batch, Scene s, Consts k,
                                                        float4* __restrict__ records, int* status_to_clear,
                                                        int* counter_to_clear, ZeroJob zero) {
  pdl_enter();
  const DevView& V = batch.v[blockIdx.y];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  prologue_clear(status_to_clear, counter_to_clear, zero);
  if (i >= V.K) return;
  float R[9], t[3];
  load_pose(s.poses, V.pose, R, t);
  const long long g = V.gauss_off + i;
  GaussRec q;
  float ml[3];
#pragma unroll
  for (int c = 0; c < 6; ++c) q.L[c] = s.chol[6 * g + c];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float oh, ol, sh, se;
    camera_centre_dd(R, t, c, oh, ol);
    two_sum(s.means[3 * g + c], -oh, sh, se);
    two_sum(sh, __fsub_rn(se, ol), q.mh[c], ml[c]);
  }
  world_record(q, ml, s.weights[g]);
  float4* r = records + kRecFloat4 * (V.rec_off + i);
  r[0] = make_float4(q.L[0], q.L[1], q.L[2], q.L[3]);
  r[1] = make_float4(q.L[4], q.L[5], q.b[0], q.b[1]);
  r[2] = make_float4(q.b[2], q.mh[0], q.mh[1], q.mh[2]);
  r[3] = make_float4(q.nbl[0], q.nbl[1], q.nbl[2], q.l2);
  if (s.crec != nullptr) {
    const float* c = s.colors + 3 * g;
    s.crec[V.rec_off + i] = make_float4(c[0], c[1], c[2], 0.f);
  }
  (void)k;
}

// The camera-plane records of a view (fmb_cam.cuh), one thread per Gaussian; the
// threads of a pair exchange halves, so that each stores 64 consecutive bytes.  The
// functions of R are those of the world-frame formulation (v = R^T c, o = -R^T t) for
// any invertible R, not only an exact rotation: A = R L and m_cam = R^-T (mu - o).
template <class B>
__global__ void __launch_bounds__(128) prologue_cam_kernel(const __grid_constant__ B batch, Scene s,
                                                            float4* __restrict__ records, int* status_to_clear,
                                                            int* counter_to_clear, ZeroJob zero) {
  pdl_enter();
  const DevView& V = batch.v[blockIdx.y];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  prologue_clear(status_to_clear, counter_to_clear, zero);
  const int Kpad = (V.K + 1) & ~1;
  if ((i & ~31) >= Kpad) return;  // whole warps only: the threads of a pair shuffle below
  const int gi = min(i, V.K - 1);
  float R[9], t[3];
  load_pose(s.poses, V.pose, R, t);
  const long long g = V.gauss_off + gi;
  const float* Lp = s.chol + 6 * g;
  const float L00 = Lp[0], L10 = Lp[1], L11 = Lp[2], L20 = Lp[3], L21 = Lp[4], L22 = Lp[5];
  FF m[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float oh, ol, sh, se;
    camera_centre_dd(R, t, c, oh, ol);
    two_sum(s.means[3 * g + c], -oh, sh, se);
    two_sum(sh, __fsub_rn(se, ol), m[c].h, m[c].l);
  }
  // R^-T = cof(R) / det(R)
  FF C[9];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int a1 = (a + 1) % 3, a2 = (a + 2) % 3, b1 = (b + 1) % 3, b2 = (b + 2) % 3;
      C[3 * a + b] = ff_prod(R[3 * a1 + b1], R[3 * a2 + b2]) - ff_prod(R[3 * a1 + b2], R[3 * a2 + b1]);
    }
  }
  const FF rdet = ff_rcp(C[0] * R[0] + C[1] * R[1] + C[2] * R[2]);
  FF mc[3], A[9];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    mc[a] = (C[3 * a] * m[0] + C[3 * a + 1] * m[1] + C[3 * a + 2] * m[2]) * rdet;
    A[3 * a + 0] = ff_prod(R[3 * a], L00) + ff_prod(R[3 * a + 1], L10) + ff_prod(R[3 * a + 2], L20);
    A[3 * a + 1] = ff_prod(R[3 * a + 1], L11) + ff_prod(R[3 * a + 2], L21);
    A[3 * a + 2] = ff_prod(R[3 * a + 2], L22);
  }
  auto P = [&](int a, int b) { return A[3 * a] * A[3 * b] + A[3 * a + 1] * A[3 * b + 1] + A[3 * a + 2] * A[3 * b + 2]; };
  const FF P00 = P(0, 0), r0 = ff_rsqrt(P00);
  const FF B00 = P00 * r0, B10 = P(1, 0) * r0, B20 = P(2, 0) * r0;
  const FF S11 = P(1, 1) - B10 * B10, r1 = ff_rsqrt(S11);
  const FF B11 = S11 * r1, B21 = (P(2, 1) - B20 * B10) * r1;
  const FF S22 = P(2, 2) - B20 * B20 - B21 * B21;
  // expansion pixel: the mean's projection, kept within an image of the view's sides
  const float z = mc[2].h;
  float pe[2];
  const float f[2] = {V.fx, V.fy}, cc[2] = {V.cx, V.cy}, side[2] = {static_cast<float>(V.W), static_cast<float>(V.H)};
  FF ce[2], rho[2];  // pe - c, and m - z c_e in pixels
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const float x = fmaf(f[c], __fdiv_rn(mc[c].h, z), cc[c]);
    // a multiple of 1/256, so that px - pe is exact
    pe[c] = 0.00390625f * rintf(256.f * (x == x ? fminf(fmaxf(x, -side[c]), 2.f * side[c]) : 0.5f * side[c]));
    ce[c] = ff_diff(pe[c], cc[c]);
    rho[c] = mc[c] * f[c] - mc[2] * ce[c];
  }
  const FF ifx = ff_rcp(FF{f[0], 0.f}), ify = ff_rcp(FF{f[1], 0.f}), sc = ff_diff(kCamScale, 0.f);
  const FF b00 = B00 * ifx * sc, b10 = B10 * ify * sc, b11 = B11 * ify * sc;
  const FF e0 = B20 * sc + b00 * ce[0] + b10 * ce[1], e1 = B21 * sc + b11 * ce[1];
  const bool real = i < V.K;
  float w[16];
  w[0] = -pe[0];
  w[1] = -pe[1];
  w[2] = b00.h;
  w[3] = b10.h;
  w[4] = z;
  w[5] = -fmaf(b00.h, rho[0].h, __fmul_rn(b10.h, rho[1].h));
  w[6] = e0.h;
  w[7] = b11.h;
  w[8] = e1.h;
  w[9] = (b11 * mc[2]).h;
  w[10] = -__fmul_rn(b11.h, rho[1].h);
  w[11] = __fmul_rn(S22.h > 0.f ? S22.h : (S22.h == S22.h ? 0.f : S22.h), kCamScale2);
  w[12] = real ? -log2f(s.weights[g]) : kDummyNl2;
  const FF m2 = P00 * P(1, 1) - P(1, 0) * P(1, 0) + P00 * P(2, 2) - P(2, 0) * P(2, 0) + P(1, 1) * P(2, 2) -
                P(2, 1) * P(2, 1);
  w[13] = __int_as_float((real ? 0 : kCamCopy) |
                         cam_flat_flags((P00 + P(1, 1) + P(2, 2)).h, m2.h, P00.h * S11.h * S22.h));
  w[14] = rho[0].h;
  w[15] = rho[1].h;
  if (s.qrec != nullptr && real) {
    // Q = B^-1 A by forward substitution (orthogonal; a row of zeros where P is singular)
    const FF r2 = ff_rsqrt(S22);
    float q[9];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const FF q0 = A[c] * r0, q1 = (A[3 + c] - B10 * q0) * r1, q2 = (A[6 + c] - B20 * q0 - B21 * q1) * r2;
      q[c] = q0.h;
      q[3 + c] = q1.h;
      q[6 + c] = q2.h;
    }
    float4* d = s.qrec + kCamQFloat4 * (static_cast<long long>(V.rec_off) + i);
    d[0] = make_float4(q[0], q[1], q[2], q[3]);
    d[1] = make_float4(q[4], q[5], q[6], q[7]);
    d[2] = make_float4(q[8], 0.f, 0.f, 0.f);
  }
  const bool odd = (i & 1) != 0;
  float rv[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) rv[k] = __shfl_xor_sync(0xffffffffu, odd ? w[k] : w[8 + k], 1);
  float cl[3] = {0.f, 0.f, 0.f}, cr[3] = {0.f, 0.f, 0.f};
  if (s.crec != nullptr) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      cl[k] = s.colors[3 * g + k];
      cr[k] = __shfl_xor_sync(0xffffffffu, cl[k], 1);
    }
  }
  if (i >= Kpad) return;
  float4* r = records + kRecFloat4 * (static_cast<long long>(V.rec_off) + i);
#pragma unroll
  for (int k = 0; k < 8; k += 2)
    r[k / 2] = odd ? make_float4(rv[k], w[8 + k], rv[k + 1], w[8 + k + 1]) : make_float4(w[k], rv[k], w[k + 1], rv[k + 1]);
  if (s.crec != nullptr)  // pair of colour records: [r r g g | b b 0 0]
    s.crec[static_cast<long long>(V.rec_off) + i] =
        odd ? make_float4(cr[2], cl[2], 0.f, 0.f) : make_float4(cl[0], cr[0], cl[1], cr[1]);
}

template <class B>
static cudaError_t launch_prologue_t(const B& b, const Scene& s, const Consts& c, float4* records, int maxK,
                                     int* status_to_clear, int* counter_to_clear, cudaStream_t st,
                                     const ZeroJob* zero) {
  dim3 grid((maxK + 127) / 128, b.n_views);
  return launch_kernel(prologue_kernel<B>, grid, dim3(128), 0, st, 1, b, s, c, records, status_to_clear,
                       counter_to_clear, zero != nullptr ? *zero : ZeroJob{});
}
cudaError_t launch_prologue(const Batch& b, const Scene& s, const Consts& c, float4* records, int maxK,
                            int* status_to_clear, int* counter_to_clear, cudaStream_t st, const ZeroJob* zero) {
  return launch_prologue_t(b, s, c, records, maxK, status_to_clear, counter_to_clear, st, zero);
}
cudaError_t launch_prologue(const BigBatch& b, const Scene& s, const Consts& c, float4* records, int maxK,
                            int* status_to_clear, int* counter_to_clear, cudaStream_t st, const ZeroJob* zero) {
  return launch_prologue_t(b, s, c, records, maxK, status_to_clear, counter_to_clear, st, zero);
}
template <class B>
static cudaError_t launch_prologue_cam_t(const B& b, const Scene& s, float4* records, int maxK, int* status_to_clear,
                                         int* counter_to_clear, cudaStream_t st, const ZeroJob* zero) {
  const dim3 grid((maxK + 1 + 127) / 128, b.n_views);
  return launch_kernel(prologue_cam_kernel<B>, grid, dim3(128), 0, st, 1, b, s, records, status_to_clear,
                       counter_to_clear, zero != nullptr ? *zero : ZeroJob{});
}
cudaError_t launch_prologue_cam(const Batch& b, const Scene& s, float4* records, int maxK, int* status_to_clear,
                                int* counter_to_clear, cudaStream_t st, const ZeroJob* zero) {
  return launch_prologue_cam_t(b, s, records, maxK, status_to_clear, counter_to_clear, st, zero);
}
cudaError_t launch_prologue_cam(const BigBatch& b, const Scene& s, float4* records, int maxK, int* status_to_clear,
                                int* counter_to_clear, cudaStream_t st, const ZeroJob* zero) {
  return launch_prologue_cam_t(b, s, records, maxK, status_to_clear, counter_to_clear, st, zero);
}

// ------------------------------------------------------------------- forward
// One ray's sums over the two Gaussians of each record, one per lane; the lanes are
// added after the last record.  Every ray constant is held in both lanes, so that a
// record's values are used as loaded (packing two rays against one Gaussian instead
// costs a move per record value).
template <bool NORMALS, bool COLOR>
struct RayAcc2 {
  f2 X, Y, K2;        // pixel centre; -(beta2 / eta) log2(e) |c|: t's share of the log2 weight
  f2 r00, r01, r11;   // NORMALS: metric of the image-plane normal components (ray_metric)
  f2 nm, Sw, Swt, Sd; // minus the running shift of the log2 weights; sums of w, w t, delta
  f2 N0, N1;          // sum w n, first two camera components over (fx, fy)
  f2 C0, C1, C2;      // COLOR: sum w c
};

// The normal g = P (t c - m) is perpendicular to the ray, so its third camera
// component is -(x g_0 + y g_1) and |g|^2 a quadratic form of the first two, written
// as (r00 h0 + r01 h1)^2 + (r11 h1)^2 for h = (g_0 / fx, g_1 / fy).
__device__ __forceinline__ void ray_metric(const DevView& V, const CamRay& r, float& r00, float& r01, float& r11) {
  const float s = fmaf(r.x, r.x, 1.0f), is = rsqrt_nr(s);
  r00 = V.fx * s * is;
  r01 = V.fy * (r.x * r.y * is);
  r11 = V.fy * (r.len * is);
}

// What a pair leaves for the sums once the shift is settled: d, the log2 weight above
// the shift, t and u.
struct FwdPair2 {
  f2 d, t, nx, u0, u1;
};
template <bool NORMALS, bool COLOR, bool FLAGGED>
__device__ __forceinline__ FwdPair2 fwd_pair2(RayAcc2<NORMALS, COLOR>& A, const CamRec2& g, f2 nB1) {
  const CamGeom2 G = cam_geom2<FLAGGED && NORMALS>(g, A.X, A.Y);
  A.Sd = add2(A.Sd, pk(ex2_approx(-lo(G.nx)), ex2_approx(-hi(G.nx))));
  return FwdPair2{fma2(G.t, A.K2, fma2(G.nx, nB1, A.nm)), G.t, G.nx, G.u0, G.u1};
}

// Raises the shift of the lane(s) whose exponent it no longer bounds.
template <bool NORMALS, bool COLOR>
__device__ __forceinline__ void fwd_raise2(RayAcc2<NORMALS, COLOR>& A, FwdPair2& q, f2 nB1) {
  const f2 e2 = fma2(q.nx, nB1, mul2(q.t, A.K2));
  float dl = lo(q.d), dh = hi(q.d), sl = 1.f, sh = 1.f, ml = lo(A.nm), mh = hi(A.nm);
  if (dl > kLazyShift) {
    sl = ex2_approx(-(lo(e2) + ml));
    ml = -lo(e2);
    dl = 0.f;
  }
  if (dh > kLazyShift) {
    sh = ex2_approx(-(hi(e2) + mh));
    mh = -hi(e2);
    dh = 0.f;
  }
  const f2 sc = pk(sl, sh);
  A.Sw = mul2(A.Sw, sc);
  A.Swt = mul2(A.Swt, sc);
  if (NORMALS) {
    A.N0 = mul2(A.N0, sc);
    A.N1 = mul2(A.N1, sc);
  }
  if (COLOR) {
    A.C0 = mul2(A.C0, sc);
    A.C1 = mul2(A.C1, sc);
    A.C2 = mul2(A.C2, sc);
  }
  A.nm = pk(ml, mh);
  q.d = pk(dl, dh);
}

template <bool NORMALS, bool COLOR>
__device__ __forceinline__ void fwd_sum2(RayAcc2<NORMALS, COLOR>& A, const CamRec2& g, const FwdPair2& q, f2 tiny, f2 c0,
                                         f2 c1, f2 c2) {
  const f2 w = ex2_2(q.d);
  A.Sw = add2(A.Sw, w);
  A.Swt = fma2(w, q.t, A.Swt);
  if (COLOR) {
    A.C0 = fma2(w, c0, A.C0);
    A.C1 = fma2(w, c1, A.C1);
    A.C2 = fma2(w, c2, A.C2);
  }
  if (NORMALS) {
    const f2 h0 = mul2(g.B00, q.u0);
    const f2 h1 = fma2(g.B11, q.u1, mul2(g.B10, q.u0));
    const f2 p0 = fma2(A.r01, h1, mul2(A.r00, h0));
    const f2 p1 = mul2(A.r11, h1);
    const f2 ws = mul2(w, rsqrt_2(fma2(p0, p0, fma2(p1, p1, tiny))));
    A.N0 = fma2(ws, h0, A.N0);
    A.N1 = fma2(ws, h1, A.N1);
  }
}

// One record against the thread's rays, with one check of the shifts for all of them (a
// check per ray cost 6 to 9 % of the kernel).  FLAGGED: a record with a flat Gaussian (with
// normals) or a copy.
template <int RPT, bool NORMALS, bool COLOR, bool FLAGGED>
__device__ __forceinline__ void fwd_record2(RayAcc2<NORMALS, COLOR> (&A)[RPT], const CamRec2& g, f2 nB1, f2 tiny, f2 c0,
                                            f2 c1, f2 c2) {
  FwdPair2 q[RPT];
#pragma unroll
  for (int r = 0; r < RPT; ++r) q[r] = fwd_pair2<NORMALS, COLOR, FLAGGED>(A[r], g, nB1);
  if (FLAGGED) {
    const bool copy = (g.flags >> 32 & kCamCopy) != 0;
#pragma unroll
    for (int r = 0; r < RPT; ++r) q[r].d = pk(lo(q[r].d), copy ? -INFINITY : hi(q[r].d));
  }
  float top = fmaxf(lo(q[0].d), hi(q[0].d));
#pragma unroll
  for (int r = 1; r < RPT; ++r) top = fmaxf(top, fmaxf(lo(q[r].d), hi(q[r].d)));
  if (top > kLazyShift) {  // rare
#pragma unroll
    for (int r = 0; r < RPT; ++r) fwd_raise2<NORMALS, COLOR>(A[r], q[r], nB1);
  }
#pragma unroll
  for (int r = 0; r < RPT; ++r) fwd_sum2<NORMALS, COLOR>(A[r], g, q[r], tiny, c0, c1, c2);
}

// A ray's sums with the two lanes brought to one shift and added.
struct RaySums {
  float m, Sw, Swt, Sd, N0, N1, C0, C1, C2;
};
template <bool NORMALS, bool COLOR>
__device__ __forceinline__ RaySums ray_sums(const RayAcc2<NORMALS, COLOR>& A) {
  RaySums r;
  const float ml = -lo(A.nm), mh = -hi(A.nm);
  r.m = fmaxf(ml, mh);
  const float sl = ex2_approx(ml - r.m), sh = ex2_approx(mh - r.m);
  r.Sw = fmaf(hi(A.Sw), sh, lo(A.Sw) * sl);
  r.Swt = fmaf(hi(A.Swt), sh, lo(A.Swt) * sl);
  r.Sd = lo(A.Sd) + hi(A.Sd);
  r.N0 = NORMALS ? fmaf(hi(A.N0), sh, lo(A.N0) * sl) : 0.f;
  r.N1 = NORMALS ? fmaf(hi(A.N1), sh, lo(A.N1) * sl) : 0.f;
  r.C0 = COLOR ? fmaf(hi(A.C0), sh, lo(A.C0) * sl) : 0.f;
  r.C1 = COLOR ? fmaf(hi(A.C1), sh, lo(A.C1) * sl) : 0.f;
  r.C2 = COLOR ? fmaf(hi(A.C2), sh, lo(A.C2) * sl) : 0.f;
  return r;
}

// The blended normal N = sum w n / sum w in the camera frame, from a ray's sums.
struct RayNormal {
  float n0, n1, n2;
};
__device__ __forceinline__ RayNormal ray_normal(const DevView& V, const RaySums& a, const CamRay& ray) {
  const float iSw = rcp_nr(a.Sw);
  const float N0 = V.fx * a.N0 * iSw, N1 = V.fy * a.N1 * iSw;
  return RayNormal{N0, N1, -fmaf(ray.x, N0, ray.y * N1)};
}

// A normal that nearly cancels (|N| below kNormalCancels, about four rays in 10 000 of
// the benchmark's scenes) has a direction that the rounding of the weights decides:
// 1e-6 in N is 1e-3 in n_f at |N| = 1e-3.  Such rays are summed again by their whole
// warp with the world-frame evaluation (pair_geom, the one the point export and the
// alpha-compositing kernels use), lane l taking Gaussians l, l + 32, ...: the normal
// there stays what that form gives, whatever the fast loop rounds.  32 Gaussians at a
// time, the shift raised at the first lane whose exponent it no longer bounds, as a
// walk in index order would.  0.1 % of the work at K = 4096.
// A ray summed again costs a warp about six times its share of the fast loop, and with
// a small beta1, where many normals are blended, |N| can be small on every ray (2048
// Gaussians of diagonal precision through a narrow field of view at beta1 = 0.1).  So a
// warp sums at most kMaxAgain of 32 rays again: where there are more, the bound on |N| is
// halved until it leaves no more than that (none after kNormalHalvings).  The others
// keep the fast loop's normal, whose N is as accurate (2.5e-7 rms in either form).  That
// scene, 8 views of 400x330: 16.4 -> 2.89 ms (2.00 without normals); at beta1 = 21.4 3.29 ->
// 2.81, and 0.90 -> 0.50 for one view, whose last warps sum no longer many rays in turn.
constexpr float kNormalCancels = 0.06f;
constexpr int kMaxAgain = 4;
constexpr int kNormalHalvings = 8;
__device__ __noinline__ RayNormal blended_normal_again(const DevView& V, const float* means, const float* chol,
                                                       const float* weights, const float* poses, float K2, float K3,
                                                       float beta1, int p) {
  const int lane = threadIdx.x & 31;
  float R[9], tp[3], vc[3], v[3], vl[3], pxy[2], oh[3], ol[3];
  load_pose(poses, V.pose, R, tp);
  pixel_ray_dd(V, R, ray_pixel(V, p), vc, v, vl, pxy);
#pragma unroll
  for (int c = 0; c < 3; ++c) camera_centre_dd(R, tp, c, oh[c], ol[c]);
  float m = -kNoShift, Sw = 0.f, N0 = 0.f, N1 = 0.f, N2 = 0.f;
  for (int base = 0; base < V.K; base += 32) {
    const bool in = base + lane < V.K;
    const long long g = V.gauss_off + min(base + lane, V.K - 1);
    GaussRec q;
    float ml[3];
#pragma unroll
    for (int c = 0; c < 6; ++c) q.L[c] = chol[6 * g + c];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float sh, se;
      two_sum(means[3 * g + c], -oh[c], sh, se);
      two_sum(sh, __fsub_rn(se, ol[c]), q.mh[c], ml[c]);
    }
    world_record(q, ml, weights[g]);
    const PairGeom G = pair_geom(q.L, q.b, q.mh, q.nbl, v[0], v[1], v[2], vl[0], vl[1], vl[2]);
    const float e2 = fmaf(fmaf(G.q, K3, q.l2), beta1, G.t * K2);
    const float g0 = q.L[0] * G.u0;
    const float g1 = fmaf(q.L[2], G.u1, q.L[1] * G.u0);
    const float g2 = fmaf(q.L[5], G.u2, fmaf(q.L[4], G.u1, q.L[3] * G.u0));
    const float rs = rsqrt_approx(fmaf(g2, g2, fmaf(g1, g1, g0 * g0)) + 1e-30f);
    auto add = [&](bool mine) {
      const float w = mine ? ex2_approx(e2 - m) : 0.f;
      const float ws = w * rs;
      Sw += w;
      N0 = fmaf(ws, g0, N0);
      N1 = fmaf(ws, g1, N1);
      N2 = fmaf(ws, g2, N2);
    };
    int start = 0;
    for (int raised = 0; raised < 32; ++raised) {  // at most one raise per lane
      const unsigned over = __ballot_sync(0xffffffffu, in && lane >= start && e2 > m + kLazyShift);
      if (over == 0) break;
      const int f = __ffs(over) - 1;
      const float mf = __shfl_sync(0xffffffffu, e2, f);
      add(in && lane >= start && lane < f);
      const float sc = ex2_approx(m - mf);
      Sw *= sc;
      N0 *= sc;
      N1 *= sc;
      N2 *= sc;
      m = mf;
      start = f;
    }
    add(in && lane >= start);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Sw += __shfl_xor_sync(0xffffffffu, Sw, o);
    N0 += __shfl_xor_sync(0xffffffffu, N0, o);
    N1 += __shfl_xor_sync(0xffffffffu, N1, o);
    N2 += __shfl_xor_sync(0xffffffffu, N2, o);
  }
  const float iSw = 1.0f / Sw;
  N0 *= iSw;
  N1 *= iSw;
  N2 *= iSw;
  return RayNormal{fmaf(R[2], N2, fmaf(R[1], N1, R[0] * N0)), fmaf(R[5], N2, fmaf(R[4], N1, R[3] * N0)),
                   fmaf(R[8], N2, fmaf(R[7], N1, R[6] * N0))};
}

// ray_normal, with the rays of the warp that need it summed again.  Whole warps call
// it; `in`: the lane has a ray (entry p of the view).
__device__ __forceinline__ RayNormal ray_normal_checked(const DevView& V, const Scene& s, const Consts& k,
                                                        const RaySums& a, const CamRay& ray, int p, bool in) {
  RayNormal N = ray_normal(V, a, ray);
  const float NN = fmaf(N.n0, N.n0, fmaf(N.n1, N.n1, N.n2 * N.n2));
  float bound = kNormalCancels * kNormalCancels;
  unsigned again = __ballot_sync(0xffffffffu, in && NN < bound);
  for (int h = 0; h < kNormalHalvings && __popc(again) > kMaxAgain; ++h) {
    bound *= 0.25f;
    again = __ballot_sync(0xffffffffu, in && NN < bound);
  }
  if (__popc(again) > kMaxAgain) again = 0;
  while (again != 0) {
    const int src = __ffs(again) - 1;
    again &= again - 1;
    const RayNormal M = blended_normal_again(V, s.means, s.chol, s.weights, s.poses, k.K2, k.K3, k.beta1,
                                             __shfl_sync(0xffffffffu, p, src));
    if ((threadIdx.x & 31) == src) N = M;
  }
  return N;
}

// Per-pixel epilogue (Eq. 3, Eq. 8, Sec. 5, Sec. 6) from a ray's sums: depth, alpha,
// the saved normalisers, the camera-frame unit normal and the flow to each target.
template <bool NORMALS, int NFLOW>
__device__ __forceinline__ void write_ray_outputs(const DevView& V, const float R[9], const float o[3],
                                                  const float (*Rj)[9], const float (*tj)[3], const bool* has_t,
                                                  const RaySums& a, const RayNormal& N, const CamRay& ray,
                                                  long long p, const FwdOut& out) {
  const int P = V.P;
  const long long off = V.pix_off;
  const float iSw = rcp_nr(a.Sw);  // Sw >= 1 / 2: the shift is one of the exponents
  const float Dz = a.Swt * iSw;
  out.depth[off + p] = Dz * ray.len;
  out.alpha[off + p] = -expm1f(-a.Sd);
  float* sv = out.saved + 3 * off;
  sv[p] = a.m + log2f(a.Sw);
  sv[P + p] = a.Sd;
  if (NORMALS) {
    const float NN = fmaf(N.n0, N.n0, fmaf(N.n1, N.n1, N.n2 * N.n2));
    const float iN = NN > 1e-37f ? rsqrt_nr(NN) : (NN == NN ? 0.f : NN);
    const float Nn = NN * iN;
    float* nrm = out.normal + 3 * off;
    nrm[p] = N.n0 * iN;
    nrm[P + p] = N.n1 * iN;
    nrm[2 * P + p] = N.n2 * iN;
    sv[2 * P + p] = Nn;
  } else {
    sv[2 * P + p] = 0.f;
  }
  if (NFLOW > 0) {
    float pt[3];  // o + R^T c Dz
#pragma unroll
    for (int k = 0; k < 3; ++k) pt[k] = fmaf(fmaf(R[k], ray.x, fmaf(R[3 + k], ray.y, R[6 + k])), Dz, o[k]);
    float* fl = out.flow + 2 * NFLOW * off;
#pragma unroll
    for (int j = 0; j < NFLOW; ++j) {
      float fu = 0.f, fv = 0.f;
      if (has_t[j]) {
        const float X0 = fmaf(Rj[j][2], pt[2], fmaf(Rj[j][1], pt[1], fmaf(Rj[j][0], pt[0], tj[j][0])));
        const float X1 = fmaf(Rj[j][5], pt[2], fmaf(Rj[j][4], pt[1], fmaf(Rj[j][3], pt[0], tj[j][1])));
        const float X2 = fmaf(Rj[j][8], pt[2], fmaf(Rj[j][7], pt[1], fmaf(Rj[j][6], pt[0], tj[j][2])));
        const float iz = 1.0f / X2;  // not rcp_nr: a point in the target's camera plane has infinite flow
        fu = fmaf(V.fx * X0, iz, V.cx) - ray.px;
        fv = fmaf(V.fy * X1, iz, V.cy) - ray.py;
      }
      fl[(2 * j) * P + p] = fu;
      fl[(2 * j + 1) * P + p] = fv;
    }
  }
}

// Shared-memory stage: kChunk records (4 float4 each), then in colour mode their
// kChunk colour records (1 float4 each).
template <bool COLOR>
__host__ __device__ constexpr int fwd_stage_float4() {
  return kChunk * (kRecFloat4 + (COLOR ? 1 : 0));
}

// Resident CTAs per SM the register budget keeps where the compiler, with the code for
// flagged records beside the plain one, would take more than 168 registers (four rays per
// thread: 220, orbit render and adjoint 661 against 654 us) or 128 (normals and flow: 157).
// The others are left alone: a bound of 4 took 128 registers instead of 118 for normals
// without flow and was slower (1023x767 at K = 333 382 against 362 us).
template <bool NORMALS, int NFLOW, int RPT, bool COLOR>
constexpr int fwd_min_blocks() {
  return COLOR ? 0 : (RPT == 4 ? 3 : (RPT == 2 && NORMALS && NFLOW > 0 ? 4 : 0));
}

template <bool NORMALS, int NFLOW, int RPT, bool COLOR = false, class B = Batch>
__global__ void __launch_bounds__(kFwdThreads, fwd_min_blocks<NORMALS, NFLOW, RPT, COLOR>())
    forward_kernel(const __grid_constant__ B batch, Scene s,
                                                              Consts k, const float4* __restrict__ records,
                                                              FwdOut out, int* status, int* counter) {
  pdl_enter();
  extern __shared__ float4 fwd_smem[];  // 1 or 2 stages x kChunk records
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ int s_item;
  const int tid = threadIdx.x;
  if (tid == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    fence_mbar_init();
  }
  __syncthreads();
  // Completed phases of each stage's barrier so far (their parity selects the next wait).
  unsigned uses0 = 0, uses1 = 0;

  for (int round = 0;; ++round) {
  const int item = next_item(counter, round, &s_item);
  if (item < 0 || item >= batch.n_items) break;
  int local;
  const int vi = find_item(batch, item, local);
  const DevView& V = batch.v[vi];
  const int P = V.P;
  // Gaussian split ks of n_gblocks (1 unless the batch is split): Gaussians
  // [ks GB, min(K, (ks + 1) GB)) of the view's object
  const int tile = local / V.n_gblocks;
  const int ks = local - tile * V.n_gblocks;
  const int kbeg = ks * V.GB;
  const int K = min(V.GB, V.K - kbeg);

  float R[9], tp[3];
  load_pose(s.poses, V.pose, R, tp);
  const float o0 = -fmaf(R[6], tp[2], fmaf(R[3], tp[1], R[0] * tp[0]));
  const float o1 = -fmaf(R[7], tp[2], fmaf(R[4], tp[1], R[1] * tp[0]));
  const float o2 = -fmaf(R[8], tp[2], fmaf(R[5], tp[1], R[2] * tp[0]));

  // Stage the first record chunks while the rays are set up.
  const float4* src = records + kRecFloat4 * (V.rec_off + kbeg);
  const int nchunks = (K + kChunk - 1) / kChunk;
  constexpr int SST = fwd_stage_float4<COLOR>();
  const float4* csrc = COLOR ? s.crec + V.rec_off + kbeg : nullptr;
  if (tid == 0) {
    for (int c = 0; c < 2 && c < nchunks; ++c) {
      const int n = (min(kChunk, K - c * kChunk) + 1) & ~1;  // whole records of two
      mbar_arrive_expect_tx(&bars[c], n * 16u * (kRecFloat4 + (COLOR ? 1 : 0)));
      bulk_g2s(fwd_smem + c * SST, src + c * kChunk * kRecFloat4, n * 16u * kRecFloat4, &bars[c]);
      if (COLOR) bulk_g2s(fwd_smem + c * SST + kChunk * kRecFloat4, csrc + c * kChunk, n * 16u, &bars[c]);
    }
  }

  RayAcc2<NORMALS, COLOR> A[RPT];
  int pix[RPT];
#pragma unroll
  for (int r = 0; r < RPT; ++r) {
    const int p = tile * (kFwdThreads * RPT) + r * kFwdThreads + tid;
    pix[r] = p;
    // rays past the end compute a valid pixel and store nothing
    const CamRay ray = cam_ray(V, ray_pixel(V, min(p, P - 1)));
    RayAcc2<NORMALS, COLOR>& a = A[r];
    a.X = dup(ray.px);
    a.Y = dup(ray.py);
    a.K2 = dup(__fmul_rn(k.K2, ray.len));
    if (NORMALS) {
      float r00, r01, r11;
      ray_metric(V, ray, r00, r01, r11);
      a.r00 = dup(r00);
      a.r01 = dup(r01);
      a.r11 = dup(r11);
    }
    a.nm = dup(kNoShift);
    a.Sw = a.Swt = a.Sd = a.N0 = a.N1 = a.C0 = a.C1 = a.C2 = dup(0.f);
  }
  const f2 nB1 = dup(-k.beta1), tiny = dup(1e-30f), zero2 = dup(0.f);
  // what takes a record through the longer code (the same for the whole CTA)
  constexpr unsigned long long kFlags = (static_cast<unsigned long long>(kCamCopy | (NORMALS ? kCamFlat : 0)) << 32) |
                                        (NORMALS ? kCamFlat : 0);

  bool failed = false;
  for (int c = 0; c < nchunks; ++c) {
    const int stage = c & 1;
    const unsigned parity = ((stage == 0 ? uses0 : uses1) + (c >> 1)) & 1u;
    const bool ok = mbar_wait_bounded(&bars[stage], parity, status);
    if (__syncthreads_or(!ok)) {
      failed = true;
      break;
    }
    const int n = min(kChunk, K - c * kChunk);
    const ulonglong2* rec = reinterpret_cast<const ulonglong2*>(fwd_smem + stage * SST);
    const ulonglong2* crs = rec + kChunk * kRecFloat4;  // colour mode: this stage's colour records
    auto color_of = [&](int i, f2& c0, f2& c1, f2& c2) {
      c0 = c1 = c2 = zero2;
      if (COLOR) {
        const ulonglong2 q0 = crs[i], q1 = crs[i + 1];
        c0 = as_f2(q0.x);
        c1 = as_f2(q0.y);
        c2 = as_f2(q1.x);
      }
    };
    int i = 0;
    while (i < n) {
      // two plain records per trip (one: 1 to 2.5 % slower), up to the first flagged one
      for (; i + 2 < n; i += 4) {
        const CamRec2 g = cam_load(rec + kRecFloat4 * i), h = cam_load(rec + kRecFloat4 * (i + 2));
        if (((g.flags | h.flags) & kFlags) != 0) break;
        f2 c0, c1, c2;
        color_of(i, c0, c1, c2);
        fwd_record2<RPT, NORMALS, COLOR, false>(A, g, nB1, tiny, c0, c1, c2);
        color_of(i + 2, c0, c1, c2);
        fwd_record2<RPT, NORMALS, COLOR, false>(A, h, nB1, tiny, c0, c1, c2);
      }
      // and then one, the last one or a flagged one or the one before it, by the longer code
      // (two at a time: 1023x767 at K = 333 370 against 366 us, K = 79 with colours 4.72
      // against 4.55 ms)
      if (i < n) {
        f2 c0, c1, c2;
        color_of(i, c0, c1, c2);
        fwd_record2<RPT, NORMALS, COLOR, true>(A, cam_load(rec + kRecFloat4 * i), nB1, tiny, c0, c1, c2);
        i += 2;
      }
    }
    __syncthreads();  // every thread is done with this stage before it is refilled
    if (tid == 0 && c + 2 < nchunks) {
      const int n2 = (min(kChunk, K - (c + 2) * kChunk) + 1) & ~1;
      mbar_arrive_expect_tx(&bars[stage], n2 * 16u * (kRecFloat4 + (COLOR ? 1 : 0)));
      if (COLOR)
        bulk_g2s(fwd_smem + stage * SST + kChunk * kRecFloat4, csrc + (c + 2) * kChunk, n2 * 16u, &bars[stage]);
      bulk_g2s(fwd_smem + stage * SST, src + (c + 2) * kChunk * kRecFloat4, n2 * 16u * kRecFloat4,
               &bars[stage]);
    }
  }
  if (failed) return;
  uses0 += (nchunks + 1) / 2;
  uses1 += nchunks / 2;

  if (V.n_gblocks > 1) {
    // Gaussian split: this split's partial sums for fwd_merge_kernel
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
      if (pix[r] >= P) continue;
      const RaySums a = ray_sums(A[r]);
      float4* q = reinterpret_cast<float4*>(out.part + V.part_off +
                                            8 * (static_cast<long long>(pix[r]) * V.n_gblocks + ks));
      q[0] = make_float4(a.m, a.Sw, a.Swt, a.Sd);
      q[1] = make_float4(a.N0, a.N1, 0.f, 0.f);
    }
    continue;
  }

  // Flow targets (uniform over the CTA).
  float Rj[NFLOW > 0 ? NFLOW : 1][9], tj[NFLOW > 0 ? NFLOW : 1][3];
  bool has_t[NFLOW > 0 ? NFLOW : 1];
#pragma unroll
  for (int j = 0; j < NFLOW; ++j) {
    const int tg = j == 0 ? V.tgt0 : V.tgt1;
    has_t[j] = tg >= 0;
    if (has_t[j]) load_pose(s.poses, tg, Rj[j], tj[j]);
  }

  const long long off = V.pix_off;
  const float o[3] = {o0, o1, o2};
#pragma unroll
  for (int r = 0; r < RPT; ++r) {
    const long long p = pix[r];
    const bool in = pix[r] < P;
    const RaySums a = ray_sums(A[r]);
    const CamRay ray = cam_ray_at(V, lo(A[r].X), lo(A[r].Y));
    RayNormal N{0.f, 0.f, 0.f};
    if (NORMALS) N = ray_normal_checked(V, s, k, a, ray, pix[r], in);
    if (!in) continue;
    if (COLOR) {
      const float iSw = rcp_nr(a.Sw);
      float* col = out.color + 3 * off;
      col[p] = a.C0 * iSw;
      col[P + p] = a.C1 * iSw;
      col[2 * P + p] = a.C2 * iSw;
    }
    write_ray_outputs<NORMALS, NFLOW>(V, R, o, Rj, tj, has_t, a, N, ray, p, out);
  }
  }  // item loop
}

static int fwd_smem_bytes(int maxK, bool color = false) {
  const int stages = maxK > kChunk ? 2 : 1;  // a second stage only when K spans several chunks
  return stages * (color ? fwd_stage_float4<true>() : fwd_stage_float4<false>()) * static_cast<int>(sizeof(float4));
}

template <bool NORMALS, int NFLOW, int RPT>
static int fwd_ctas_per_sm_t(int maxK) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, forward_kernel<NORMALS, NFLOW, RPT>, kFwdThreads,
                                                    fwd_smem_bytes(maxK)) != cudaSuccess)
    return 1;
  return n > 0 ? n : 1;
}

template <bool NORMALS, int NFLOW, int RPT, bool COLOR = false, class B>
static cudaError_t launch_fwd_t(const B& b, const Scene& s, const Consts& c, const float4* records,
                                const FwdOut& o, int maxK, int* status, int* counter, cudaStream_t st) {
  auto kern = forward_kernel<NORMALS, NFLOW, RPT, COLOR, B>;
  const int smem = fwd_smem_bytes(maxK, COLOR);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  int grid = b.n_items;
  if (counter) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    grid = std::min(b.n_items, std::max(1, sms) * fwd_ctas_per_sm_t<NORMALS, NFLOW, RPT>(maxK));
  }
  return launch_kernel(kern, dim3(grid), dim3(kFwdThreads), smem, st, 1, b, s, c, records, o, status, counter);
}

template <bool NORMALS, int NFLOW, class B>
static cudaError_t launch_fwd_r(int rpt, const B& b, const Scene& s, const Consts& c, const float4* records,
                                const FwdOut& o, int maxK, int* status, int* counter, cudaStream_t st) {
  if (o.color != nullptr)  // colour mode: two rays per thread only
    return launch_fwd_t<NORMALS, NFLOW, 2, true>(b, s, c, records, o, maxK, status, counter, st);
  switch (rpt) {
    case 1: return launch_fwd_t<NORMALS, NFLOW, 1>(b, s, c, records, o, maxK, status, counter, st);
    case 2: return launch_fwd_t<NORMALS, NFLOW, 2>(b, s, c, records, o, maxK, status, counter, st);
    default: return launch_fwd_t<NORMALS, NFLOW, 4>(b, s, c, records, o, maxK, status, counter, st);
  }
}

template <class B>
static cudaError_t launch_forward_t(const B& b, const Scene& s, const Consts& c, const float4* records,
                                    bool normals, int n_flow, int rpt, int maxK, const FwdOut& o, int* status,
                                    int* counter, cudaStream_t st) {
  if (normals) {
    if (n_flow == 0) return launch_fwd_r<true, 0>(rpt, b, s, c, records, o, maxK, status, counter, st);
    if (n_flow == 1) return launch_fwd_r<true, 1>(rpt, b, s, c, records, o, maxK, status, counter, st);
    return launch_fwd_r<true, 2>(rpt, b, s, c, records, o, maxK, status, counter, st);
  }
  if (n_flow == 0) return launch_fwd_r<false, 0>(rpt, b, s, c, records, o, maxK, status, counter, st);
  if (n_flow == 1) return launch_fwd_r<false, 1>(rpt, b, s, c, records, o, maxK, status, counter, st);
  return launch_fwd_r<false, 2>(rpt, b, s, c, records, o, maxK, status, counter, st);
}
cudaError_t launch_forward(const Batch& b, const Scene& s, const Consts& c, const float4* records, bool normals,
                           int n_flow, int rpt, int maxK, const FwdOut& o, int* status, int* counter,
                           cudaStream_t st) {
  return launch_forward_t(b, s, c, records, normals, n_flow, rpt, maxK, o, status, counter, st);
}
cudaError_t launch_forward(const BigBatch& b, const Scene& s, const Consts& c, const float4* records, bool normals,
                           int n_flow, int rpt, int maxK, const FwdOut& o, int* status, int* counter,
                           cudaStream_t st) {
  return launch_forward_t(b, s, c, records, normals, n_flow, rpt, maxK, o, status, counter, st);
}

int forward_rays_per_cta(int rpt) { return kFwdThreads * rpt; }

// ------------------------------------------------ merge of a Gaussian-split forward
// One thread per ray.  Each split left its max-shifted sums (m_s, Sw_s, Swt_s, Sd_s,
// N_s); brought to the largest shift m they add exactly like the terms of one pass:
// Sw = sum_s 2^(m_s - m) Sw_s (likewise Swt and N), Sd = sum_s Sd_s.  The epilogue
// then writes the planes as the unsplit forward does.
constexpr int kMergeThreads = 128;
int forward_merge_rays_per_item() { return kMergeThreads; }

template <bool NORMALS, int NFLOW, class B>
__global__ void __launch_bounds__(kMergeThreads) fwd_merge_kernel(const __grid_constant__ B batch, Scene s,
                                                                  Consts c, FwdOut out) {
  pdl_enter();
  int local;
  const int vi = find_item(batch, blockIdx.x, local);
  const DevView& V = batch.v[vi];
  const int P = V.P;
  const bool in = local * kMergeThreads + static_cast<int>(threadIdx.x) < P;
  // threads past the end merge a valid ray and store nothing
  const long long p = min(local * kMergeThreads + static_cast<int>(threadIdx.x), P - 1);
  float R[9], tp[3];
  load_pose(s.poses, V.pose, R, tp);
  const float o[3] = {-fmaf(R[6], tp[2], fmaf(R[3], tp[1], R[0] * tp[0])),
                      -fmaf(R[7], tp[2], fmaf(R[4], tp[1], R[1] * tp[0])),
                      -fmaf(R[8], tp[2], fmaf(R[5], tp[1], R[2] * tp[0]))};
  float Rj[NFLOW > 0 ? NFLOW : 1][9], tj[NFLOW > 0 ? NFLOW : 1][3];
  bool has_t[NFLOW > 0 ? NFLOW : 1];
#pragma unroll
  for (int j = 0; j < NFLOW; ++j) {
    const int tg = j == 0 ? V.tgt0 : V.tgt1;
    has_t[j] = tg >= 0;
    if (has_t[j]) load_pose(s.poses, tg, Rj[j], tj[j]);
  }
  const CamRay ray = cam_ray(V, ray_pixel(V, static_cast<int>(p)));
  const int S = V.S;  // splits of this view
  const float4* q = reinterpret_cast<const float4*>(out.part + V.part_off + 8 * p * S);
  float m = -INFINITY;
  for (int k = 0; k < S; ++k) m = fmaxf(m, q[2 * k].x);
  RaySums a{m, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int k = 0; k < S; ++k) {
    const float4 q0 = q[2 * k], q1 = q[2 * k + 1];
    const float sc = ex2_approx(q0.x - m);
    a.Sw = fmaf(sc, q0.y, a.Sw);
    a.Swt = fmaf(sc, q0.z, a.Swt);
    a.Sd += q0.w;
    if (NORMALS) {
      a.N0 = fmaf(sc, q1.x, a.N0);
      a.N1 = fmaf(sc, q1.y, a.N1);
    }
  }
  RayNormal N{0.f, 0.f, 0.f};
  if (NORMALS) N = ray_normal_checked(V, s, c, a, ray, static_cast<int>(p), in);
  if (in) write_ray_outputs<NORMALS, NFLOW>(V, R, o, Rj, tj, has_t, a, N, ray, p, out);
}

template <class B>
static cudaError_t launch_forward_merge_t(const B& b, const Scene& s, const Consts& c, bool normals, int n_flow, const FwdOut& o,
                                          cudaStream_t st) {
  if (b.n_items <= 0) return cudaSuccess;
  const dim3 grid(b.n_items), block(kMergeThreads);
  if (normals) {
    if (n_flow == 0) return launch_kernel(fwd_merge_kernel<true, 0, B>, grid, block, 0, st, 1, b, s, c, o);
    if (n_flow == 1) return launch_kernel(fwd_merge_kernel<true, 1, B>, grid, block, 0, st, 1, b, s, c, o);
    return launch_kernel(fwd_merge_kernel<true, 2, B>, grid, block, 0, st, 1, b, s, c, o);
  }
  if (n_flow == 0) return launch_kernel(fwd_merge_kernel<false, 0, B>, grid, block, 0, st, 1, b, s, c, o);
  if (n_flow == 1) return launch_kernel(fwd_merge_kernel<false, 1, B>, grid, block, 0, st, 1, b, s, c, o);
  return launch_kernel(fwd_merge_kernel<false, 2, B>, grid, block, 0, st, 1, b, s, c, o);
}
cudaError_t launch_forward_merge(const Batch& b, const Scene& s, const Consts& c, bool normals, int n_flow,
                                 const FwdOut& o, cudaStream_t st) {
  return launch_forward_merge_t(b, s, c, normals, n_flow, o, st);
}
cudaError_t launch_forward_merge(const BigBatch& b, const Scene& s, const Consts& c, bool normals, int n_flow,
                                 const FwdOut& o, cudaStream_t st) {
  return launch_forward_merge_t(b, s, c, normals, n_flow, o, st);
}

int forward_ctas_per_sm(bool normals, int n_flow, int rpt, int maxK) {
  (void)normals;
  (void)n_flow;
  switch (rpt) {
    case 1: return fwd_ctas_per_sm_t<true, 1, 1>(maxK);
    case 2: return fwd_ctas_per_sm_t<true, 1, 2>(maxK);
    default: return fwd_ctas_per_sm_t<true, 1, 4>(maxK);
  }
}

}  // namespace fmb
