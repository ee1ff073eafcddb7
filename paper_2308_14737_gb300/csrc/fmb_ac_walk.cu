// fmb_ac_walk.cu -- forward of the alpha-compositing variant (Sec. 3.3, Eq. 9-10) for
// batches of whole images with many rays: one thread per ray instead of one warp.
//
// The weights w_i = T_i (1 - e^-delta_i) need the hits of a ray in depth order.  A
// thread takes a column of `run` pixels, top to bottom, and keeps its depth order in
// shared memory (one byte per Gaussian): the order of the pixel above, which differs
// from the current one by a few neighbours that change places.  It walks that order
// once, evaluating each hit and passing it through a window of kWindow hits sorted in
// registers: what leaves the window is blended at once -- transmittance, weight and
// sums advance hit by hit, without scans, shuffles or a reduction -- and written back
// as the new order.  A hit that would have to move by more than the window leaves it
// out of order; such rays are sorted by the whole warp, one after the other, and the
// warp walks once more.  (Walking again from the order just written until every ray's
// depths ascend took up to 20 times the warp-per-ray kernel's time on small images of
// many Gaussians, 2.5 times on one 631x473 view at K = 256: 3.27 -> 0.65 ms.)  Hits at exactly equal depth share the sum in front of their run
// (the indicator of Eq. 10 is strict).  Every pair's depth comes from pair_geom, as in
// the warp-per-ray kernels, so that orders and ties are the same bits.
//
// The first pixel of a column starts from a warp's bitonic sort of a ray at most four
// pixels away (four sorts per warp).
//
// Bound by its instructions (76 % of the issue rate, the compares and selects of the
// window half of them; 562 warp instructions per ray with normals against the warp-per-ray
// kernel's 1225).  Orbit of 16 views 320x240, K = 100, depth, alpha and flow: 1.340 -> 0.699
// ms; with normals 1.452 -> 0.848 ms.
#include <algorithm>

#include "fmb_ac.cuh"
#include "fmb_ac_walk.cuh"
#include "fmb_internal.cuh"

namespace fmb {

constexpr int kWalkThreads = 128;
constexpr int kWindow = 7;  // 6, 8 and 11: 2 to 6 % slower on the orbit (more walks, more compares)
constexpr int kRing = kWindow + 1;  // slots of a thread's pair values: one per hit in the window and the new one
constexpr int kWalkMaxRun = 32;

// one_minus_exp_neg with its series in Horner form (7 operations; a walk is bound by
// its instruction count).
__device__ __forceinline__ float walk_one_minus_exp_neg(float x) {
  float p = fmaf(x, 1.f / 5040.f, -1.f / 720.f);
  p = fmaf(x, p, 1.f / 120.f);
  p = fmaf(x, p, -1.f / 24.f);
  p = fmaf(x, p, 1.f / 6.f);
  p = fmaf(x, p, -0.5f);
  p = fmaf(x, p, 1.f);
  return x < 0.25f ? x * p : 1.f - ex2_approx(-x * kLog2e);
}

// Bytes of a thread's order: 4 x odd, so that the threads of a warp read and write
// their bytes in 32 different banks.
__host__ __device__ constexpr int walk_row_bytes(int maxK) { return 4 * (((maxK + 3) / 4) | 1); }

// The ring holds a pair's density (and normal) while its hit is in the window.
template <bool NORMALS>
__host__ __device__ constexpr int walk_ring_float4() {
  return (NORMALS ? 4 : 1) * kRing * kWalkThreads / 4;
}

int ac_walk_threads() { return kWalkThreads; }
// Column length: the longest power of two up to 32 that leaves every SM 1536 columns
// (two rounds of resident CTAs, which evens out the columns that walk more often), at
// least 2; 0 (the warp-per-ray kernel) when that leaves fewer than 640 columns per SM.
// 16 x 320x240 at K = 100: 384 / 768 / 1536 / 3000 columns per SM asked for 1081 / 932 /
// 858 / 930 us (measured before the loop was split and unrolled); 631x473 at K = 61, one
// round of columns of 2: 160 us against the warp kernel's 215.
// 0 also where the warp-per-ray kernel, which refines the previous pixel's order, is as
// fast.  Hits change places in proportion to K / f from one pixel to the next (f: focal
// length in pixels), and a sort costs about K log^2 K, so that the limit is on K^2 / f;
// a launch (at most 64 views) needs 448 columns of 2 per SM.  Time of this kernel over
// the warp kernel's, scenes of random / diagonal precisions:
//   fewer columns: 210 per SM, K = 40 / 100 1.15 / 1.57, 0.83 / 1.55; 51 (800 views of 16x16) 1.2 to 2.1
//   505 to 1580 columns, K^2 / f: K = 40 53 0.62 / 0.53, 125 0.90 / 0.81; K = 100 16 0.76 / 0.78, 78 1.00 /
//     0.78, 100 0.97 / 0.80, 156 1.19 / 0.98; K = 160 80 0.90 / 0.66, 200 1.20 / 0.98; K = 256 105 1.39 / 0.99
//   2590 and 4040 columns: K = 100 156 0.68 / 0.56; K = 160 250 0.69 / 0.60, 400 0.93 / 0.69; K = 256 64 0.96 /
//     0.70, 205 1.33 / 1.01
int ac_walk_run(long long total_rays, int launches, int maxK, float min_f, int sms) {
  const long long sm = std::max(sms, 1);
  int run = kWalkMaxRun;
  while (run > 2 && total_rays < 1536 * sm * run) run >>= 1;
  if (total_rays < 640 * sm * run) return 0;
  const long long rays = total_rays / std::max(launches, 1);
  if (rays < 448 * sm * 2) return 0;
  const float limit = maxK <= 192 && rays >= 2000 * sm * 2 ? 400.f : (maxK <= 64 ? 128.f : 100.f);
  return static_cast<float>(maxK) * static_cast<float>(maxK) > limit * min_f ? 0 : run;
}

template <bool NORMALS, int NFLOW, int M>
__global__ void __launch_bounds__(kWalkThreads) forward_ac_walk_kernel(const __grid_constant__ Batch batch, Scene s,
                                                                       Consts k, const float4* __restrict__ records,
                                                                       FwdOut out, int run, int row_bytes,
                                                                       int* counter) {
  pdl_enter();
  // ring [1 or 4][kRing][threads] floats | records [K][kAcRecStride float4] | orders [threads][row_bytes]
  extern __shared__ float4 walk_smem[];
  __shared__ int s_item;
  const int tid = threadIdx.x, lane = tid & 31;
  float* ring = reinterpret_cast<float*>(walk_smem) + tid;
  float4* srec = walk_smem + walk_ring_float4<NORMALS>();
  for (int round = 0;; ++round) {
    const int item = next_item(counter, round, &s_item);
    if (item < 0 || item >= batch.n_items) break;
    int tile;
    const int vi = find_item(batch, item, tile);
    const DevView& V = batch.v[vi];
    const int P = V.P, K = V.K, W = V.W;
    unsigned char* orders = reinterpret_cast<unsigned char*>(srec + kAcRecStride * K);
    unsigned char* ord = orders + tid * row_bytes;
    if (round > 0) __syncthreads();  // the previous item's records are dead
    ac_stage_records(srec, records + kRecFloat4 * V.rec_off, K);
    float R[9], tp[3];
    load_pose(s.poses, V.pose, R, tp);
    const long long off = V.pix_off;
    const float4* crec = s.crec != nullptr && out.color != nullptr ? s.crec + V.rec_off : nullptr;
    // column u of the view: x = u mod W in the strip of `run` rows u / W
    const int columns = W * ((V.H + run - 1) / run);
    const int u = min(tile * kWalkThreads + tid, columns - 1);
    const bool live = tile * kWalkThreads + tid < columns;
    const int strip = u / W;
    const int p_first = strip * run * W + (u - strip * W);

    // Rays to sort before the next walk, and the rows of the warp that take a sorted order:
    // first the starting orders.
    unsigned todo = 0x10101010u;
    int spread = 8;

#pragma unroll 1
    for (int j = 0; j < run; ++j) {
      const int p = p_first + j * W;
      const bool in = live && p < P;
      if (!__any_sync(kFull, in)) break;
      float vc[3], v[3], vl[3], pxy[2];
      pixel_ray_dd(V, R, min(p, P - 1), vc, v, vl, pxy);
      float Sd = 0.f, Ws = 0.f, WT = 0.f, WN0 = 0.f, WN1 = 0.f, WN2 = 0.f, WC0 = 0.f, WC1 = 0.f, WC2 = 0.f;
      for (int walk = 0; walk < 2; ++walk) {
#pragma unroll 1
        for (unsigned left = todo; left != 0; left &= left - 1) {
          const int src = __ffs(left) - 1;
          float sc[3], sv[3], sl[3], sxy[2];
          pixel_ray_dd(V, R, __shfl_sync(kFull, min(p, P - 1), src), sc, sv, sl, sxy);
          unsigned long long key[M];
#pragma unroll
          for (int m = 0; m < M; ++m) {
            const int e = (m << 5) | lane;
            key[m] = kNoKey;
            if (e < K) {
              const AcPair q = ac_pair_eval<false>(srec + kAcRecStride * e, sv, sl, k);
              key[m] = (static_cast<unsigned long long>(order_bits(fminf(q.t, INFINITY))) << 32) | static_cast<unsigned>(e);
            }
          }
          warp_bitonic_sort<M>(key, lane);
          unsigned char* rows = orders + ((tid & ~31) + (src & ~(spread - 1))) * row_bytes;
#pragma unroll
          for (int m = 0; m < M; ++m)
            if (lane * M + m < K)
              for (int r = 0; r < spread; ++r) rows[r * row_bytes + lane * M + m] = static_cast<unsigned char>(key[m]);
        }
        todo = 0;
        spread = 1;
        __syncwarp();
        // the window: ascending depths, each with its Gaussian and ring slot (e | slot << 8)
        float wt[kWindow];
        int wi[kWindow];
#pragma unroll
        for (int l = 0; l < kWindow; ++l) {
          wt[l] = -INFINITY;
          wi[l] = 0;
        }
        float last = -INFINITY, front = 0.f;
        bool ascending = true;
        int free_slot = 0;  // ring slot of the next hit: the first kWindow + 1 in turn, then the one last left
        Sd = Ws = WT = WN0 = WN1 = WN2 = WC0 = WC1 = WC2 = 0.f;
        // one step: hit i of the order enters the window (load), the smallest leaves (emit)
        auto step = [&](int i, bool load, bool emit) {
          float xt = INFINITY;
          int xi = 0;
          if (load) {
            const int e = ord[i], slot = free_slot;
            const AcPair q = ac_pair_eval<NORMALS>(srec + kAcRecStride * e, v, vl, k);
            xt = fminf(q.t, INFINITY);  // a NaN depth (invalid data) must not lose its place in the order
            xi = e | (slot << 8);
            ring[slot * kWalkThreads] = q.dl;
            if (NORMALS) {
#pragma unroll
              for (int c = 0; c < 3; ++c) ring[((c + 1) * kRing + slot) * kWalkThreads] = q.n[c];
            }
          }
          // the smallest of the window and x leaves; x takes its place among the rest
          // (after equal depths)
          bool after[kWindow + 1];
#pragma unroll
          for (int l = 0; l < kWindow; ++l) after[l] = !(xt < wt[l]);
          after[kWindow] = false;
          const float t_out = fminf(xt, wt[0]);
          const int i_out = after[0] ? wi[0] : xi;
#pragma unroll
          for (int l = 0; l < kWindow; ++l) {
            wi[l] = l + 1 < kWindow && after[l + 1] ? wi[l + 1 < kWindow ? l + 1 : l] : (after[l] ? xi : wi[l]);
            wt[l] = l + 1 < kWindow ? fmaxf(wt[l], fminf(xt, wt[l + 1 < kWindow ? l + 1 : l])) : fmaxf(wt[l], xt);
          }
          if (!emit) {
            free_slot = i + 1;
            return;
          }
          const int e = i_out & 255, slot = i_out >> 8;
          free_slot = slot;  // for the next hit
          ord[i - kWindow] = static_cast<unsigned char>(e);
          const float dl = ring[slot * kWalkThreads];
          ascending = ascending && !(t_out < last);
          if (t_out != last) front = Sd;  // a run of equal depths shares the sum in front of it
          last = t_out;
          const float w = ex2_approx(-front * kLog2e) * walk_one_minus_exp_neg(dl);
          Sd += dl;
          Ws += w;
          WT = fmaf(w, t_out, WT);
          if (NORMALS) {
            WN0 = fmaf(w, ring[(kRing + slot) * kWalkThreads], WN0);
            WN1 = fmaf(w, ring[(2 * kRing + slot) * kWalkThreads], WN1);
            WN2 = fmaf(w, ring[(3 * kRing + slot) * kWalkThreads], WN2);
          }
          if (crec != nullptr) {
            const float4 c = __ldg(crec + e);
            WC0 = fmaf(w, c.x, WC0);
            WC1 = fmaf(w, c.y, WC1);
            WC2 = fmaf(w, c.z, WC2);
          }
        };
        for (int i = 0; i < kWindow; ++i) step(i, i < K, false);
#pragma unroll 2
        for (int i = kWindow; i < K; ++i) step(i, true, true);
        for (int i = max(K, kWindow); i < K + kWindow; ++i) step(i, false, true);
        const unsigned late = __ballot_sync(kFull, in && !ascending);
        if (late == 0 || walk > 0) break;  // the second walk is over sorted or ascending orders
        todo = late;
      }

      if (in) {
        if (out.order != nullptr) {
          // 16 bytes at a time; the row of the workspace holds 32 M bytes
          uint4* dst = reinterpret_cast<uint4*>(out.order + (off + p) * (32 * M));
          const unsigned* w4 = reinterpret_cast<const unsigned*>(ord);
          const int words = row_bytes / 4;
          for (int q = 0; 16 * q < K; ++q) {
            uint4 o;
            o.x = w4[4 * q];
            o.y = w4[min(4 * q + 1, words - 1)];
            o.z = w4[min(4 * q + 2, words - 1)];
            o.w = w4[min(4 * q + 3, words - 1)];
            dst[q] = o;
          }
        }
        const float iW = Ws > 0.f ? 1.0f / Ws : 0.f;
        const float D = WT * iW;
        if (crec != nullptr) {
          float* col = out.color + 3 * off;
          col[p] = WC0 * iW;
          col[P + p] = WC1 * iW;
          col[2 * P + p] = WC2 * iW;
        }
        out.depth[off + p] = D;
        out.alpha[off + p] = -expm1f(-Sd);
        float* sv = out.saved + 3 * off;
        sv[p] = Ws;
        sv[P + p] = Sd;
        if (NORMALS) {
          const float N0 = WN0 * iW, N1 = WN1 * iW, N2 = WN2 * iW;
          const float Nn = sqrtf(fmaf(N0, N0, fmaf(N1, N1, N2 * N2)));
          const float iN = Nn > 0.f ? 1.0f / Nn : 0.f;
          const float n0 = N0 * iN, n1 = N1 * iN, n2 = N2 * iN;
          float* nrm = out.normal + 3 * off;
          nrm[p] = fmaf(R[2], n2, fmaf(R[1], n1, R[0] * n0));
          nrm[P + p] = fmaf(R[5], n2, fmaf(R[4], n1, R[3] * n0));
          nrm[2 * P + p] = fmaf(R[8], n2, fmaf(R[7], n1, R[6] * n0));
          sv[2 * P + p] = Nn;
        } else {
          sv[2 * P + p] = 0.f;
        }
        if (NFLOW > 0) {
          const float o0 = -fmaf(R[6], tp[2], fmaf(R[3], tp[1], R[0] * tp[0]));
          const float o1 = -fmaf(R[7], tp[2], fmaf(R[4], tp[1], R[1] * tp[0]));
          const float o2 = -fmaf(R[8], tp[2], fmaf(R[5], tp[1], R[2] * tp[0]));
          const float p0 = fmaf(v[0], D, o0), p1 = fmaf(v[1], D, o1), p2 = fmaf(v[2], D, o2);
          float* fl = out.flow + 2 * NFLOW * off;
#pragma unroll
          for (int f = 0; f < NFLOW; ++f) {
            const int tg = f == 0 ? V.tgt0 : V.tgt1;
            float fu = 0.f, fv = 0.f;
            if (tg >= 0) {
              float Rj[9], tj[3];
              load_pose(s.poses, tg, Rj, tj);
              const float X0 = fmaf(Rj[2], p2, fmaf(Rj[1], p1, fmaf(Rj[0], p0, tj[0])));
              const float X1 = fmaf(Rj[5], p2, fmaf(Rj[4], p1, fmaf(Rj[3], p0, tj[1])));
              const float X2 = fmaf(Rj[8], p2, fmaf(Rj[7], p1, fmaf(Rj[6], p0, tj[2])));
              const float iz = 1.0f / X2;
              fu = fmaf(V.fx * X0, iz, V.cx) - pxy[0];
              fv = fmaf(V.fy * X1, iz, V.cy) - pxy[1];
            }
            fl[(2 * f) * P + p] = fu;
            fl[(2 * f + 1) * P + p] = fv;
          }
        }
      }
    }
  }
}

template <bool NORMALS, int NFLOW, int M>
static cudaError_t launch_walk_t(const Batch& b, const Scene& s, const Consts& c, const float4* records, int maxK,
                                 const FwdOut& o, int run, int* counter, cudaStream_t st) {
  auto kern = forward_ac_walk_kernel<NORMALS, NFLOW, M>;
  const int row = walk_row_bytes(maxK);
  const int smem = walk_ring_float4<NORMALS>() * 16 + maxK * kAcRecStride * 16 + kWalkThreads * row;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  int grid = b.n_items;
  if (counter) {
    int dev = 0, sms = 0, per = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kWalkThreads, smem);
    grid = std::min(b.n_items, std::max(1, sms) * std::max(1, per));
  }
  return launch_kernel(kern, dim3(grid), dim3(kWalkThreads), smem, st, 1, b, s, c, records, o, run, row, counter);
}

template <bool NORMALS, int NFLOW>
static cudaError_t launch_walk_m(const Batch& b, const Scene& s, const Consts& c, const float4* records, int maxK,
                                 const FwdOut& o, int run, int* counter, cudaStream_t st) {
  switch (ac_lanes_per_ray_elements(maxK)) {
    case 2: return launch_walk_t<NORMALS, NFLOW, 2>(b, s, c, records, maxK, o, run, counter, st);
    case 4: return launch_walk_t<NORMALS, NFLOW, 4>(b, s, c, records, maxK, o, run, counter, st);
    default: return launch_walk_t<NORMALS, NFLOW, 8>(b, s, c, records, maxK, o, run, counter, st);
  }
}

cudaError_t launch_forward_ac_walk(const Batch& b, const Scene& s, const Consts& c, const float4* records, bool normals,
                                   int n_flow, int maxK, const FwdOut& o, int run, int* counter, cudaStream_t st) {
  if (run < 1 || run > kWalkMaxRun) return cudaErrorInvalidValue;
  if (normals) {
    if (n_flow == 0) return launch_walk_m<true, 0>(b, s, c, records, maxK, o, run, counter, st);
    if (n_flow == 1) return launch_walk_m<true, 1>(b, s, c, records, maxK, o, run, counter, st);
    return launch_walk_m<true, 2>(b, s, c, records, maxK, o, run, counter, st);
  }
  if (n_flow == 0) return launch_walk_m<false, 0>(b, s, c, records, maxK, o, run, counter, st);
  if (n_flow == 1) return launch_walk_m<false, 1>(b, s, c, records, maxK, o, run, counter, st);
  return launch_walk_m<false, 2>(b, s, c, records, maxK, o, run, counter, st);
}

}  // namespace fmb
