// REINFORCE backward of the network in FP32 (Eq. 10): the gradient of
//   sum_b w_b log q(s_b),   w_b = -(l_b - mean l) / (beta B),
// by a teacher-forced forward and hand-written backward, in two kernels:
//   bwd32_delta_kernel  per 32 samples: hidden values, dX and the deltas, all
//                       layers in one CTA, written unit-major for the next
//   bwd32_wgrad_kernel  per 64 x 64 block of a weight matrix and slice of the
//                       batch: sum_b delta[b][m] act[b][n] and the bias sums
// Both are bound by the FP32 pipe (about 28 k and 23 k live multiply-adds per
// sample for the 64-128-128-64 network).  One kernel that kept a chunk's
// weight gradient in global memory and added to it every 32 samples, with one
// output per thread, took 1.51 ms for 5 x 16,384 samples of that network;
// these two take 0.28 + 0.15 ms (0.35 + 0.15 with streamed weights; the
// multiply-adds alone take 0.11).  For small networks one kernel
// (bwd32_small_kernel) is the faster form and stays.
#include <math.h>

#include <type_traits>

#include "common.cuh"

namespace tnvan {

#define B3_TS 32   // samples per CTA of the delta kernel
#define B3_TP 36   // row stride of its [unit][sample] tiles (16-byte rows, 8 lanes x 16 bytes conflict-free)
#define B3_MB 128  // output units per block
#define B3_KC 32   // inputs per weight stage
#define B3_WS (B3_MB * B3_TP)  // floats of a weight stage ([unit][36], or transposed [input][132])
#define B3_WT (B3_MB + 4)

namespace {

// Rows of the per-instance workspace, unit-major [unit][ldb]: S, A1, A2, dX, dA2, dA1.
struct Rows {
  float *S, *A1, *A2, *X, *dA2, *dA1;
};
__device__ __forceinline__ Rows rows_of(const MadeDev& md, float* w, long long ldb) {
  Rows r;
  r.S = w;
  r.A1 = r.S + md.D * ldb;
  r.A2 = r.A1 + md.H1 * ldb;
  r.X = r.A2 + md.H2 * ldb;
  r.dA2 = r.X + md.D * ldb;
  r.dA1 = r.dA2 + md.H2 * ldb;
  return r;
}

// Inputs of packed output row o of layer l: a prefix of this length (rows are
// sorted by degree, so it does not decrease with o).
__device__ __forceinline__ int fan_in(const MadeDev& md, int l, int o) {
  if (l == md.nh) return md.nh == 0 ? o : (md.nh == 1 ? md.c1 : md.c2)[o];
  const int d = md.layer[l].deg_out[o];
  return l == 0 ? d : md.c1[d];
}
// First output row of layer l + 1 that reads packed unit j of hidden layer l.
__device__ __forceinline__ int fan_out0(const MadeDev& md, int l, int j) {
  const int d = md.layer[l].deg_out[j];
  return l + 1 == md.nh ? d : md.c2[d - 1];
}

__device__ __forceinline__ void cp_async(float* dst, const float* src, int vec, bool on) {
  if (vec == 4)  // a constant once inlined
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(on ? 16 : 0)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(on ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Rounds a row length up to a whole number of 8 x 16-byte chunks (the swizzle's period).
__host__ __device__ __forceinline__ int res_cols(int n) { return (n + 31) & ~31; }

// The weights of a layer as a half-CTA reads them.  RES: the whole matrix in
// shared memory, row r at base + r * cols, 16-byte chunk q at q ^ ((r >> 2) & 7)
// (four lanes four rows apart then hit four different bank groups, in the
// forward product and in the transposed one).  Otherwise 128-unit x 32-input
// stages are fetched into a two-slot ring as they are used.
struct Weights {
  const float* W;     // global [rows][cols]
  const float* res;   // shared copy (RES)
  int rows, cols, vec;
};

// Fetch stage c of output block o0: forward as [128 units][36], transposed as
// [32 inputs][132]; zeros outside W.
template <bool FWD>
__device__ __forceinline__ void fetch(const Weights& w, float* dst, int o0, int c, int tid) {
  const int r0 = FWD ? o0 : c * B3_KC, c0 = FWD ? c * B3_KC : o0;
  constexpr int LD = FWD ? B3_TP : B3_WT, NR = FWD ? B3_MB : B3_KC;
  auto run = [&](auto v) {
    constexpr int V = decltype(v)::value, LN = (FWD ? B3_KC : B3_MB) / V, RS = 256 / LN;  // lanes a row, rows a pass
    const int cc = (tid % LN) * V, r = tid / LN;
    const bool con = c0 + cc < w.cols;
    const float* src = w.W + (long long)(r0 + r) * w.cols + c0 + cc;
    float* d = dst + r * LD + cc;
#pragma unroll
    for (int j = 0; j < NR / RS; ++j) {
      const bool on = con && r0 + r + j * RS < w.rows;
      cp_async(d + j * RS * LD, on ? src + (long long)j * RS * w.cols : w.W, V, on);
    }
  };
  if (w.vec == 4) run(std::integral_constant<int, 4>());
  else run(std::integral_constant<int, 1>());
}

// Barrier of the 256 threads that share a tile.
template <bool RES>
__device__ __forceinline__ void tile_sync(int half) {
  if (RES) asm volatile("bar.sync %0, 256;" ::"r"(1 + half) : "memory");
  else __syncthreads();
}

enum { B3_RELU, B3_DX };

// One forward layer on the tile: out[o][t] = epi(bias[o] + sum_{j < fan_in(o)} W[o][j] in[j][t]).
// A thread holds 4 rows x 4 samples; per output four partial sums over j mod 4
// for the multiples of four, the remaining inputs on the first, added as
// (a0 + a1) + (a2 + a3).  That order is part of the result: a unit whose
// pre-activation is within rounding of 0 has its ReLU decided by it.
template <bool RES, int EPI>
__device__ __forceinline__ void forward_layer(const Weights& wt, const int* fan, const float* in, float* out,
                                              float* gout, long long ldb, float* wst, const float* wb, int tid,
                                              int half) {
  const int M = wt.rows;
  const float* bias = wt.W + (long long)M * wt.cols;
  const int w = tid >> 5, lt = tid & 7, lo = (tid >> 3) & 3;
  // 16-row groups in an order that gives the four schedulers equal sums of fan-ins
  const int grp = w < 4 ? w : 11 - w;
  for (int o0 = 0; o0 < M; o0 += B3_MB) {
    const int c1 = RES ? 1 : (fan[min(M, o0 + B3_MB) - 1] + B3_KC - 1) / B3_KC;
    const int base = o0 + 16 * grp + 4 * lo;
    int n[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) n[j] = fan[min(base + j, M - 1)];
    const bool live = o0 + 16 * grp < M;  // per warp
    float a[4][4][4];  // [row][sample][j mod 4]
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int q = 0; q < 4; ++q) a[j][t][q] = 0.f;
    if (!RES) {
      if (c1 > 0) fetch<true>(wt, wst, o0, 0, tid);
      cp_commit();
    }
    for (int c = 0; c < c1; ++c) {
      if (!RES) {
        if (c + 1 < c1) fetch<true>(wt, wst + ((c + 1) & 1) * B3_WS, o0, c + 1, tid);
        cp_commit();
        cp_wait<1>();
        __syncthreads();
      }
      const int k0 = RES ? 0 : c * B3_KC, k1 = RES ? n[3] : k0 + B3_KC;
      // rows past M (RES: no such rows in memory) read the last one; their results are dropped
      const float* wp[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        wp[j] = RES ? wt.res + min(base + j, M - 1) * res_cols(wt.cols)
                    : wst + (c & 1) * B3_WS + (base - o0 + j) * B3_TP;
      const int swz = (base >> 2) & 7, swl = ((M - 1) >> 2) & 7;
      auto wq = [&](int j, int k) {
        if (RES) return *reinterpret_cast<const float4*>(wp[j] + ((((k >> 2) ^ (base + j < M ? swz : swl))) << 2));
        return *reinterpret_cast<const float4*>(wp[j] + (k - k0));
      };
      if (live) {
        const float* xp = in + k0 * B3_TP + 4 * lt;
        int k = k0;
        const int kfull = min(k1, n[0] & ~3), kend = min(k1, n[3]);
#pragma unroll 1
        for (; k < kfull; k += 4, xp += 4 * B3_TP) {  // all four rows connected
          float4 x[4], ww[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) x[q] = *reinterpret_cast<const float4*>(xp + q * B3_TP);
#pragma unroll
          for (int j = 0; j < 4; ++j) ww[j] = wq(j, k);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float wv[4] = {ww[j].x, ww[j].y, ww[j].z, ww[j].w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              a[j][0][q] = fmaf(wv[q], x[q].x, a[j][0][q]);
              a[j][1][q] = fmaf(wv[q], x[q].y, a[j][1][q]);
              a[j][2][q] = fmaf(wv[q], x[q].z, a[j][2][q]);
              a[j][3][q] = fmaf(wv[q], x[q].w, a[j][3][q]);
            }
          }
        }
        // the rows' ends: a whole quad to the four sums, fewer inputs to the first
#pragma unroll 1
        for (; k < kend; k += 4, xp += 4 * B3_TP) {
          float4 x[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) x[q] = *reinterpret_cast<const float4*>(xp + q * B3_TP);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float4 ww = wq(j, k);
            const float wv[4] = {ww.x, ww.y, ww.z, ww.w};
            const int rest = n[j] - k;
            if (rest >= 4) {
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                a[j][0][q] = fmaf(wv[q], x[q].x, a[j][0][q]);
                a[j][1][q] = fmaf(wv[q], x[q].y, a[j][1][q]);
                a[j][2][q] = fmaf(wv[q], x[q].z, a[j][2][q]);
                a[j][3][q] = fmaf(wv[q], x[q].w, a[j][3][q]);
              }
            } else {
#pragma unroll
              for (int q = 0; q < 3; ++q) {
                if (q >= rest) break;
                a[j][0][0] = fmaf(wv[q], x[q].x, a[j][0][0]);
                a[j][1][0] = fmaf(wv[q], x[q].y, a[j][1][0]);
                a[j][2][0] = fmaf(wv[q], x[q].z, a[j][2][0]);
                a[j][3][0] = fmaf(wv[q], x[q].w, a[j][3][0]);
              }
            }
          }
        }
      }
      if (!RES) __syncthreads();
    }
    if (live) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int o = base + j;
        if (o >= M) continue;
        const float b = __ldg(bias + o);
        float r[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const float x = b + ((a[j][t][0] + a[j][t][1]) + (a[j][t][2] + a[j][t][3]));
          if (EPI == B3_RELU) {
            r[t] = fmaxf(x, 0.f);
          } else {
            // d log q / d x = s sigmoid(-s x); S of this entry is read before dX replaces it
            const float s = out ? out[o * B3_TP + 4 * lt + t] : in[o * B3_TP + 4 * lt + t];
            r[t] = wb[4 * lt + t] * s / (1.f + expf(s * x));
          }
        }
        const float4 v = make_float4(r[0], r[1], r[2], r[3]);
        if (out) *reinterpret_cast<float4*>(out + o * B3_TP + 4 * lt) = v;
        *reinterpret_cast<float4*>(gout + o * ldb + 4 * lt) = v;
      }
    }
  }
  tile_sync<RES>(half);
}

// Delta of a hidden layer from the layer above (dn [row][t], weights wt), in
// place of the layer's own values h: h[j][t] = 1[h > 0] sum_{i >= first(j)} dn[i][t] W[i][j].
template <bool RES>
__device__ __forceinline__ void delta_layer(const Weights& wt, const int* first, const float* dn, float* h,
                                            float* gout, long long ldb, float* wst, int tid, int half) {
  const int M = wt.cols, K = wt.rows;
  const int w = tid >> 5, lt = tid & 7, lo = (tid >> 3) & 3;
  const int grp = w < 4 ? w : 11 - w;
  for (int o0 = 0; o0 < M; o0 += B3_MB) {
    const int c0 = RES ? 0 : first[o0] / B3_KC, c1 = RES ? 1 : (K + B3_KC - 1) / B3_KC;
    const int base = o0 + 16 * grp + 4 * lo;
    int f[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) f[j] = first[min(base + j, M - 1)];
    const bool live = o0 + 16 * grp < M;
    float a[4][4][2];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int t = 0; t < 4; ++t) a[j][t][0] = a[j][t][1] = 0.f;
    if (!RES) {
      if (c0 < c1) fetch<false>(wt, wst + (c0 & 1) * B3_WS, o0, c0, tid);
      cp_commit();
    }
    for (int c = c0; c < c1; ++c) {
      if (!RES) {
        if (c + 1 < c1) fetch<false>(wt, wst + ((c + 1) & 1) * B3_WS, o0, c + 1, tid);
        cp_commit();
        cp_wait<1>();
        __syncthreads();
      }
      if (live) {
        const int k0 = RES ? 0 : c * B3_KC, k1 = RES ? K : min(k0 + B3_KC, K);
        const float* ws = wst + (c & 1) * B3_WS + (base - o0);
        auto wq = [&](int k) {
          // a row is res_cols long, so a thread past M reads inside it
          if (RES) return *reinterpret_cast<const float4*>(wt.res + k * res_cols(M) + (((base >> 2) ^ ((k >> 2) & 7)) << 2));
          return *reinterpret_cast<const float4*>(ws + (k - k0) * B3_WT);
        };
        auto step = [&](int k, int p) {
          const float4 x = *reinterpret_cast<const float4*>(dn + k * B3_TP + 4 * lt);
          const float4 q = wq(k);
          const float wv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            a[j][0][p] = fmaf(wv[j], x.x, a[j][0][p]);
            a[j][1][p] = fmaf(wv[j], x.y, a[j][1][p]);
            a[j][2][p] = fmaf(wv[j], x.z, a[j][2][p]);
            a[j][3][p] = fmaf(wv[j], x.w, a[j][3][p]);
          }
        };
        int k = max(k0, f[0]);
#pragma unroll 1
        for (; k < min(k1, f[3]); ++k) {  // the rows' first connections
          const float4 x = *reinterpret_cast<const float4*>(dn + k * B3_TP + 4 * lt);
          const float4 q = wq(k);
          const float wv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (k < f[j]) continue;
            a[j][0][0] = fmaf(wv[j], x.x, a[j][0][0]);
            a[j][1][0] = fmaf(wv[j], x.y, a[j][1][0]);
            a[j][2][0] = fmaf(wv[j], x.z, a[j][2][0]);
            a[j][3][0] = fmaf(wv[j], x.w, a[j][3][0]);
          }
        }
#pragma unroll 2
        for (; k + 2 <= k1; k += 2) {
          step(k, 0);
          step(k + 1, 1);
        }
        if (k < k1) step(k, 0);
      }
      if (!RES) __syncthreads();
    }
    if (live) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int o = base + j;
        if (o >= M) continue;
        float4* hp = reinterpret_cast<float4*>(h + o * B3_TP + 4 * lt);
        const float4 hv = *hp;
        const float4 v = make_float4(hv.x > 0.f ? a[j][0][0] + a[j][0][1] : 0.f,
                                     hv.y > 0.f ? a[j][1][0] + a[j][1][1] : 0.f,
                                     hv.z > 0.f ? a[j][2][0] + a[j][2][1] : 0.f,
                                     hv.w > 0.f ? a[j][3][0] + a[j][3][1] : 0.f);
        *hp = v;
        *reinterpret_cast<float4*>(gout + o * ldb + 4 * lt) = v;
      }
    }
  }
  tile_sync<RES>(half);
}

}  // namespace

// Floats of the resident copy of an instance's weights.
int bwd32_res_floats(int D, int nh, int H1, int H2) {
  if (nh == 0) return D * res_cols(D);
  if (nh == 1) return H1 * res_cols(D) + D * res_cols(H1);
  return H1 * res_cols(D) + H2 * res_cols(H1) + D * res_cols(H2);
}
// Dynamic shared memory of the delta kernel for max_units = D + H1 + H2 and
// res weight floats (0: streamed weights).
int bwd32_smem_bytes(int max_units, int res) {
  const int tile = B3_TS + (max_units + 3) * B3_TP;  // 1 / b weights, then the units; three rows are read past the last
  return 4 * (2 * max_units + 3 + (res ? res + 2 * tile : 2 * B3_WS + tile));
}

// 256 threads per tile of 32 samples: thread = 4 samples (8 lanes) x 4 units (4
// lanes), a warp 16 units, 128 units a pass.  Per 64 FMAs a thread reads eight
// 16-byte shared words, each one conflict-free wavefront per warp, so the FMA
// pipe has twice the shared-memory time.
// RES (the weights fit beside two tiles): one CTA per SM holds its instance's
// weights for all its tiles, two halves of 256 threads each on tiles of their
// own, li.tile_begin counting CTAs.  Otherwise one tile per CTA, li.tile_begin
// counting tiles, with the weights streamed through shared memory: each stage
// costs two barriers and its copies' latency.
template <bool RES>
__global__ void __launch_bounds__(RES ? 512 : 256, RES ? 1 : 2)
    bwd32_delta_kernel(const InstDev* __restrict__ inst, const LaunchInfo li, const Bwd32Ws bw,
                       const int8_t* __restrict__ spins, const double* __restrict__ logZR,
                       const float* __restrict__ logq, const double* __restrict__ stats) {
  extern __shared__ __align__(16) float sm[];
  const int k = find_inst(li, blockIdx.x);
  const InstDev& I = inst[k];
  const MadeDev& md = I.made;
  const int D = md.D, nh = md.nh, H1 = md.H1, H2 = md.H2;
  const int half = RES ? threadIdx.x >> 8 : 0, tid = threadIdx.x & 255;
  const int units = D + H1 + H2;
  int* fan = reinterpret_cast<int*>(sm);  // fan-ins: layer 0, 1 (hidden), output
  int* first = fan + units;               // first connections: hidden layer 0, 1
  float* tile = sm + ((2 * units + 3) & ~3);
  float* wst = tile;
  Weights wt[3];
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    if (l > nh) break;
    const LayerDev& L = md.layer[l];
    wt[l].W = md.packed + L.dst_off;
    wt[l].rows = L.nout;
    wt[l].cols = L.nin;
    wt[l].vec = ((L.nin & 3) == 0 && (reinterpret_cast<uintptr_t>(wt[l].W) & 15) == 0) ? 4 : 1;
    wt[l].res = nullptr;
    if (RES) {
      float* dst = tile;
      const int cp = res_cols(L.nin);
      for (int e = threadIdx.x; e < L.nout * cp; e += 512) {
        const int r = e / cp, c = e - r * cp;
        dst[r * cp + ((((c >> 2) ^ ((r >> 2) & 7)) << 2) | (c & 3))] =
            c < L.nin ? wt[l].W[(long long)r * L.nin + c] : 0.f;
      }
      wt[l].res = dst;
      tile += L.nout * cp;
    }
  }
  if (!RES) tile += 2 * B3_WS;
  int* fl[3] = {fan, nh >= 1 ? fan + H1 : fan, nh >= 2 ? fan + H1 + H2 : fan + H1};
  for (int l = 0; l <= nh; ++l)
    for (int o = threadIdx.x; o < md.layer[l].nout; o += blockDim.x) {
      fl[l][o] = fan_in(md, l, o);
      if (l < nh) first[(l ? H1 : 0) + o] = fan_out0(md, l, o);
    }
  tile += half * (B3_TS + (units + 3) * B3_TP);
  float* wb = tile;  // [32]
  float* S = wb + B3_TS;
  float* A1 = S + D * B3_TP;
  float* A2 = A1 + H1 * B3_TP;  // three rows past each are readable (the last quad of a fan-in)
  __syncthreads();
  const int ntile = (bw.nb + B3_TS - 1) / B3_TS;
  const int rank = blockIdx.x - li.tile_begin[k], nblk = li.tile_begin[k + 1] - li.tile_begin[k];
  const double wscale = -1.0 / (li.beta[k] * stats_batch(stats + 8 * k));
  for (int it = RES ? 2 * rank + half : rank; it < ntile; it += RES ? 2 * nblk : ntile) {
    const long long b0 = bw.b0 + (long long)it * B3_TS;
    const Rows g = rows_of(md, bw.base + bw.off[k] + (long long)it * B3_TS, bw.ldb);
    const int nv = min(B3_TS, bw.nb - it * B3_TS);
    if (tid < B3_TS) {
      const long long o = (long long)k * li.batch + b0 + tid;
      wb[tid] = tid < nv ? (float)(wscale * (logZR[o] - (double)logq[o] - stats[8 * k + 4])) : 0.f;
    }
    const int8_t* sp = spins + I.spin_units * li.batch + b0 * D;
    for (int t = tid >> 5; t < B3_TS; t += 8)
      for (int i = tid & 31; i < D; i += 32) S[i * B3_TP + t] = t < nv ? (float)sp[(long long)t * D + i] : 0.f;
    tile_sync<RES>(half);
    for (int e = tid; e < D * 8; e += 256)
      *reinterpret_cast<float4*>(g.S + (long long)(e >> 3) * bw.ldb + 4 * (e & 7)) =
          *reinterpret_cast<const float4*>(S + (e >> 3) * B3_TP + 4 * (e & 7));
    if (nh >= 1) forward_layer<RES, B3_RELU>(wt[0], fl[0], S, A1, g.A1, bw.ldb, wst, wb, tid, half);
    if (nh >= 2) forward_layer<RES, B3_RELU>(wt[1], fl[1], A1, A2, g.A2, bw.ldb, wst, wb, tid, half);
    // dX replaces S (its last readers were the first layer's); without hidden layers S is the input
    if (nh == 0) forward_layer<RES, B3_DX>(wt[0], fl[0], S, nullptr, g.X, bw.ldb, wst, wb, tid, half);
    else if (nh == 1) forward_layer<RES, B3_DX>(wt[1], fl[1], A1, S, g.X, bw.ldb, wst, wb, tid, half);
    else forward_layer<RES, B3_DX>(wt[2], fl[2], A2, S, g.X, bw.ldb, wst, wb, tid, half);
    if (nh == 2) {
      delta_layer<RES>(wt[2], first + H1, S, A2, g.dA2, bw.ldb, wst, tid, half);
      delta_layer<RES>(wt[1], first, A2, A1, g.dA1, bw.ldb, wst, tid, half);
    } else if (nh == 1) {
      delta_layer<RES>(wt[1], first, S, A1, g.dA1, bw.ldb, wst, tid, half);
    }
  }
}

// 128 threads per 64 x 64 block (8 lanes x 8 rows, 16 groups x 4 columns, both
// interleaved so that 16-byte reads along the samples are conflict-free), the
// slice's samples 32 at a time through a two-stage cp.async ring.  Products of
// 32 samples are summed first and then added to the running sum.  Blocks
// wholly outside the MADE mask are left out (their entries are never read).
__global__ void __launch_bounds__(128, 4) bwd32_wgrad_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
                                                             const Bwd32Ws bw, int splits, int rows, int row0,
                                                             float* __restrict__ partials, long long part_stride) {
  __shared__ __align__(16) float As[2][64 * B3_TP], Bs[2][64 * B3_TP];
  const int k = blockIdx.z;
  if ((li.skip[k >> 5] >> (k & 31)) & 1u) return;
  const MadeDev& md = inst[k].made;
  // this CTA's layer and block
  int l = 0, blk = blockIdx.x, nt = 0;
  for (; l <= md.nh; ++l) {
    nt = (md.layer[l].nin + 63) >> 6;
    const int cnt = ((md.layer[l].nout + 63) >> 6) * nt;
    if (blk < cnt) break;
    blk -= cnt;
  }
  if (l > md.nh) return;
  const int M = md.layer[l].nout, N = md.layer[l].nin;
  const int m0 = (blk / nt) << 6, n0 = (blk % nt) << 6;
  if (n0 > 0 && fan_in(md, l, min(m0 + 64, M) - 1) <= n0) return;
  const long long ldb = bw.ldb;
  const Rows g = rows_of(md, bw.base + bw.off[k], ldb);
  const float* A = (l == md.nh ? g.X : (l == 1 ? g.dA2 : g.dA1)) + m0 * ldb;
  const float* Bm = (l == 0 ? g.S : (l == 1 ? g.A1 : g.A2)) + n0 * ldb;
  const int per = (int)((ldb / 32 + splits - 1) / splits);
  const int c_lo = blockIdx.y * per, c_hi = min((int)(ldb / 32), c_lo + per);
  const int tid = threadIdx.x, ml = tid & 7, ng = tid >> 3;
  auto stage = [&](int c) {
    float *a = As[c & 1], *b = Bs[c & 1];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = ng + 16 * j, q = ml * 4;
      const bool ma = m0 + r < M, nb = n0 + r < N;
      cp_async(a + r * B3_TP + q, ma ? A + r * ldb + 32ll * c + q : A, 4, ma);
      cp_async(b + r * B3_TP + q, nb ? Bm + r * ldb + 32ll * c + q : Bm, 4, nb);
    }
  };
  float acc[8][4], bsum = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  if (c_lo < c_hi) stage(c_lo);
  cp_commit();
  for (int c = c_lo; c < c_hi; ++c) {
    if (c + 1 < c_hi) stage(c + 1);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
    const float *a = As[c & 1], *b = Bs[c & 1];
    float p[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) p[i][j] = 0.f;
#pragma unroll 2
    for (int t = 0; t < 32; t += 4) {
      float4 bv[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) bv[j] = *reinterpret_cast<const float4*>(b + (ng + 16 * j) * B3_TP + t);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 av = *reinterpret_cast<const float4*>(a + (ml + 8 * i) * B3_TP + t);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          p[i][j] = fmaf(av.x, bv[j].x, p[i][j]);
          p[i][j] = fmaf(av.y, bv[j].y, p[i][j]);
          p[i][j] = fmaf(av.z, bv[j].z, p[i][j]);
          p[i][j] = fmaf(av.w, bv[j].w, p[i][j]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] += p[i][j];
    if (n0 == 0 && tid < 64) {  // the bias: row sums of the deltas
      float s = 0.f;
#pragma unroll
      for (int t = 0; t < 32; t += 4) {
        const float4 v = *reinterpret_cast<const float4*>(a + tid * B3_TP + t);
        s += v.x;
        s += v.y;
        s += v.z;
        s += v.w;
      }
      bsum += s;
    }
    __syncthreads();
  }
  float* G = partials + ((long long)k * rows + row0 + blockIdx.y) * part_stride + md.layer[l].dst_off;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = m0 + ml + 8 * i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + ng + 16 * j;
      if (n < N) G[(long long)m * N + n] = acc[i][j];
    }
  }
  if (n0 == 0 && tid < 64 && m0 + tid < M) G[(long long)M * N + m0 + tid] = bsum;
}

// ---------------------------------------------------------------------------
// Small networks: all of it in one kernel, a chunk of li.tile samples per CTA, 32
// at a time, a warp's lanes on the samples and the warps on the units; the
// chunk's weight gradient is kept in the CTA's row of `partials`, in L2.  What
// bounds it is the chain of barriers between the layers; the two kernels above
// add a launch and the rows' way through memory, which such a network's few
// multiply-adds do not repay (us here and there): one 5-16 network, 250 samples
// 25 and 33; five over 64,000 samples of 5 units and no hidden layer 172 and 228,
// of 5-16 281 and 394, of 40-17-9 (1,259 parameters) 524 and 597.  Above that
// the wide layers lose at large batches what the launch gains at small ones:
// 40 units and no hidden layer (1,640) 25 and 31 at 60 samples, 365 and 324 at
// 5 x 64,000; 1-32-48 (1,697) 621 and 504.  The outer product stays a function
// with a loop of four samples a turn: unrolled in place it took 106 registers and
// 20 to 25 % more time.
// Forward sums as forward_layer adds them; per weight the sum over 32 samples,
// added to the chunk's.
// ---------------------------------------------------------------------------
namespace {

constexpr int SM_TP = 33;  // row stride of its [unit][sample] tiles

__device__ __forceinline__ float small_dot(const float* __restrict__ w, const float* col, int n) {
  float a[4] = {0.f, 0.f, 0.f, 0.f};
  int j = 0;
  for (; j + 4 <= n; j += 4)
#pragma unroll
    for (int p = 0; p < 4; ++p) a[p] = fmaf(__ldg(w + j + p), col[(j + p) * SM_TP], a[p]);
  for (; j < n; ++j) a[0] = fmaf(__ldg(w + j), col[j * SM_TP], a[0]);
  return (a[0] + a[1]) + (a[2] + a[3]);
}

// sum_{i = i0}^{n-1} col[i] w[i * stride]
__device__ __forceinline__ float small_dot_t(const float* __restrict__ w, int stride, const float* col, int i0, int n) {
  float a0 = 0.f, a1 = 0.f;
  int i = i0;
  for (; i + 2 <= n; i += 2) {
    a0 = fmaf(__ldg(w + i * stride), col[i * SM_TP], a0);
    a1 = fmaf(__ldg(w + (i + 1) * stride), col[(i + 1) * SM_TP], a1);
  }
  if (i < n) a0 = fmaf(__ldg(w + i * stride), col[i * SM_TP], a0);
  return a0 + a1;
}

// G[m][n] (+)= sum_t delta[m][t] act[n][t], and the bias sums after it; 4 x 4 weights a thread.
__device__ __noinline__ void small_outer(float* __restrict__ G, const float* delta, const float* act, int M, int N,
                                         bool first) {
  const int mb = (M + 3) >> 2, nb = (N + 3) >> 2;
  for (int blk = threadIdx.x; blk < mb * nb; blk += blockDim.x) {
    const int m0 = (blk / nb) << 2, n0 = (blk % nb) << 2;
    float acc[4][4] = {};
#pragma unroll 4
    for (int t = 0; t < B3_TS; ++t) {
      float a[4], b[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) a[r] = m0 + r < M ? delta[(m0 + r) * SM_TP + t] : 0.f;
#pragma unroll
      for (int c = 0; c < 4; ++c) b[c] = n0 + c < N ? act[(n0 + c) * SM_TP + t] : 0.f;
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(a[r], b[c], acc[r][c]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (m0 + r < M && n0 + c < N) {
          float* g = G + (m0 + r) * N + n0 + c;
          *g = first ? acc[r][c] : *g + acc[r][c];
        }
  }
  float* gb = G + M * N;
  for (int m = threadIdx.x; m < M; m += blockDim.x) {
    float sum = 0.f;
#pragma unroll 4
    for (int t = 0; t < B3_TS; ++t) sum += delta[m * SM_TP + t];
    gb[m] = first ? sum : gb[m] + sum;
  }
}

}  // namespace

__global__ void __launch_bounds__(256)
    bwd32_small_kernel(const InstDev* __restrict__ inst, const LaunchInfo li, const int8_t* __restrict__ spins,
                       const double* __restrict__ logZR, const float* __restrict__ logq,
                       const double* __restrict__ stats, float* __restrict__ partials, long long part_stride) {
  extern __shared__ __align__(16) float sm[];
  const int k = find_inst(li, blockIdx.x);
  const InstDev& I = inst[k];
  const MadeDev& md = I.made;
  const int D = md.D, nh = md.nh, H1 = md.H1, H2 = md.H2;
  const int tid = threadIdx.x, nth = blockDim.x, t = tid & 31, q = tid >> 5, nq = nth >> 5;
  float* S = sm;  // spins, hidden values, dX and the deltas
  float* A1 = S + D * SM_TP;
  float* A2 = A1 + H1 * SM_TP;
  float* X = A2 + H2 * SM_TP;
  float* dA2 = X + D * SM_TP;
  float* dA1 = dA2 + H2 * SM_TP;
  const float *last = nh == 0 ? S : (nh == 1 ? A1 : A2), *W1 = md.packed + md.layer[0].dst_off;
  const float* W2 = nh >= 2 ? md.packed + md.layer[1].dst_off : nullptr;
  const float *Wo = md.packed + md.layer[nh].dst_off, *b1 = W1 + H1 * D, *b2 = W2 + H2 * H1, *bo = Wo + D * md.Hl;
  const int* deg1 = nh >= 1 ? md.layer[0].deg_out : nullptr;
  const int* deg2 = nh >= 2 ? md.layer[1].deg_out : nullptr;
  const int Hl = md.Hl;
  const int *c1 = md.c1, *c2 = md.c2, *cl = nh == 1 ? c1 : c2;
  const double wscale = -1.0 / (li.beta[k] * stats_batch(stats + 8 * k)), mean = stats[8 * k + 4];
  float* G = partials + (long long)blockIdx.x * part_stride;
  float *G1 = G + md.layer[0].dst_off, *Go = G + md.layer[nh].dst_off;
  float* G2 = nh >= 2 ? G + md.layer[1].dst_off : nullptr;
  const int8_t* sp = spins + I.spin_units * li.batch;
  const int chunk = li.tile, b_lo = (blockIdx.x - li.tile_begin[k]) * chunk, n = min(li.batch - b_lo, chunk);
  for (int c = 0; c < n; c += B3_TS) {
    const int b0 = b_lo + c, nv = min(B3_TS, n - c);
    for (int e = tid; e < B3_TS * D; e += nth) {
      const int tt = e / D, i = e - tt * D;
      S[i * SM_TP + tt] = tt < nv ? (float)sp[(long long)b0 * D + e] : 0.f;
    }
    __syncthreads();
    if (nh >= 1) {
      for (int o = q; o < H1; o += nq)
        A1[o * SM_TP + t] = fmaxf(__ldg(b1 + o) + small_dot(W1 + o * D, S + t, deg1[o]), 0.f);
      __syncthreads();
    }
    if (nh >= 2) {
      for (int o = q; o < H2; o += nq)
        A2[o * SM_TP + t] = fmaxf(__ldg(b2 + o) + small_dot(W2 + o * H1, A1 + t, c1[deg2[o]]), 0.f);
      __syncthreads();
    }
    const long long at = (long long)k * li.batch + b0 + t;
    const float wb = t < nv ? (float)(wscale * (logZR[at] - (double)logq[at] - mean)) : 0.f;
    for (int i = q; i < D; i += nq) {
      const float x = __ldg(bo + i) + small_dot(Wo + i * Hl, last + t, nh == 0 ? i : cl[i]), sv = S[i * SM_TP + t];
      X[i * SM_TP + t] = wb * sv / (1.f + expf(sv * x));
    }
    __syncthreads();
    if (nh >= 2) {
      for (int o = q; o < H2; o += nq)
        dA2[o * SM_TP + t] = A2[o * SM_TP + t] > 0.f ? small_dot_t(Wo + o, Hl, X + t, deg2[o], D) : 0.f;
      __syncthreads();
      for (int j = q; j < H1; j += nq)
        dA1[j * SM_TP + t] = A1[j * SM_TP + t] > 0.f ? small_dot_t(W2 + j, H1, dA2 + t, c2[deg1[j] - 1], H2) : 0.f;
      __syncthreads();
    } else if (nh == 1) {
      for (int j = q; j < H1; j += nq)
        dA1[j * SM_TP + t] = A1[j * SM_TP + t] > 0.f ? small_dot_t(Wo + j, Hl, X + t, deg1[j], D) : 0.f;
      __syncthreads();
    }
    small_outer(Go, X, last, D, Hl, c == 0);
    if (nh >= 2) small_outer(G2, dA2, A1, H2, H1, c == 0);
    if (nh >= 1) small_outer(G1, dA1, S, H1, D, c == 0);
    __syncthreads();  // tiles free for the next samples
  }
}

int bwd32_small_smem(int max_units) { return 2 * max_units * SM_TP * (int)sizeof(float); }

cudaError_t launch_bwd32_small(const InstDev* d_inst, const LaunchInfo& li, int smem, const int8_t* spins,
                               const double* logZR, const float* logq, const double* stats, float* partials,
                               long long part_stride, cudaStream_t s) {
  const int nblk = li.tile_begin[li.n_inst];
  if (nblk == 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(bwd32_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  bwd32_small_kernel<<<nblk, 256, smem, s>>>(d_inst, li, spins, logZR, logq, stats, partials, part_stride);
  return cudaGetLastError();
}

cudaError_t launch_bwd32_delta(const InstDev* d_inst, const LaunchInfo& li, const Bwd32Ws& bw, bool resident, int smem,
                               const int8_t* spins, const double* logZR, const float* logq, const double* stats,
                               cudaStream_t s) {
  const int nblk = li.tile_begin[li.n_inst];
  if (nblk == 0) return cudaSuccess;
  void (*kern)(const InstDev*, const LaunchInfo, const Bwd32Ws, const int8_t*, const double*, const float*,
               const double*) = resident ? bwd32_delta_kernel<true> : bwd32_delta_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  kern<<<nblk, resident ? 512 : 256, smem, s>>>(d_inst, li, bw, spins, logZR, logq, stats);
  return cudaGetLastError();
}

cudaError_t launch_bwd32_wgrad(const InstDev* d_inst, const LaunchInfo& li, const Bwd32Ws& bw, int max_blocks,
                               int splits, int rows, int row0, float* partials, long long part_stride,
                               cudaStream_t s) {
  if (li.n_inst == 0 || max_blocks == 0) return cudaSuccess;
  bwd32_wgrad_kernel<<<dim3(max_blocks, splits, li.n_inst), 128, 0, s>>>(d_inst, li, bw, splits, rows, row0, partials,
                                                                        part_stride);
  return cudaGetLastError();
}

}  // namespace tnvan
