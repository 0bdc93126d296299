// Hidden values, dX and deltas of the BF16 REINFORCE backward (Eq. 10) on
// tcgen05, for networks the fused kernel (k_bwd_fused.cu) does not take: up to
// two hidden layers and D of at most 256 units each.
//
// One CTA (512 threads) takes 128 samples through every layer:
//   A1 = relu(S W1^T + b1), A2 = relu(A1 W2^T + b2),
//   dX = w s sigmoid(-s (A2 Wo^T + bo)),
//   dA2 = (dX Wo) 1[A2 > 0], dA1 = (dA2 W2) 1[A1 > 0],
// each rounded to BF16 as the next product's operand and kept in shared memory
// (K-major core matrices; dX takes S's place, dA2 A2's and dA1 A1's); each
// tile, and S, is copied out as it stands by one bulk copy, for the weight
// gradients below.  Weights are the packed BF16 tiles (MadeDev::ctiles): one
// copy serves the forward product (K-major) and the transposed one (MN-major),
// 32 inputs a stage, by bulk copies through a ring that runs ahead across
// products.  Warp 0 issues copies and MMAs; accumulators in TMEM, K in steps of
// 16 in input order; 16 warps share each epilogue (a quarter of the columns
// each).  Bound by latency: five dependent products of 1 to 8 stages, each with
// an epilogue.  The 48-256-256-48 network with 3 x 4,096 samples took 134 us as
// five GEMM launches (64 columns a CTA, operands through global memory) after
// one for the weights and spins, 73 us with weights fetched and rows stored by
// the threads (129,000 warp instructions a CTA), 50 us in this form.
#include <cuda_bf16.h>

#include "common.cuh"
#include "tc.cuh"

namespace tnvan {

#define BC_THREADS 512

namespace {

__host__ __device__ __forceinline__ int r16(int n) { return (n + 15) & ~15; }

// Byte offset of element (row r, column k) of a K-major operand of kp columns.
__device__ __forceinline__ uint32_t k_off(int r, int k, int kp) { return tc::kmajor_off(r, k, kp * 2, 2); }

// Shared -> global bulk copy as a group of its own; wait until every group's
// source has been read.
__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// One product of the chain, from the weight tile [rp][cp] (padded widths) at
// element `off` of the network's tiles: forward N = rp, K = cp; transposed
// N = cp, K = rp.
struct Prod {
  int off, rp, cp, tr;
  __device__ int N() const { return tr ? cp : rp; }
  __device__ int K() const { return tr ? rp : cp; }
};

// Stage ks (32 inputs) of a product's weights into dst by the lanes of warp 0:
// forward [row group][4 core matrices], transposed [4 row groups][core matrices].
__device__ __forceinline__ void fetch(const Prod& p, int ks, const uint16_t* tiles, unsigned char* dst, uint64_t* bar,
                                      int lane) {
  const int g0 = 4 * ks, ng = min(4, (p.K() >> 3) - g0);  // 8-input groups
  const uint32_t bytes = p.tr ? 16u * (uint32_t)(ng * p.cp) : 128u * (uint32_t)ng;  // a copy's
  if (lane == 0) mbar_expect_tx(bar, p.tr ? bytes : bytes * (uint32_t)(p.rp >> 3));
  __syncwarp();
  const uint16_t* src = tiles + p.off;
  if (p.tr) {
    if (lane == 0) bulk_g2s(dst, src + g0 * 8 * p.cp, bytes, bar);
  } else if (lane < (p.rp >> 3)) {
    bulk_g2s(dst + 512 * lane, src + lane * 8 * p.cp + g0 * 64, bytes, bar);
  }
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 x = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&x);
}
__device__ __forceinline__ float bf_lo(uint32_t x) { return __uint_as_float(x << 16); }
__device__ __forceinline__ float bf_hi(uint32_t x) { return __uint_as_float(x & 0xFFFF0000u); }

}  // namespace

// Shared memory: the tile's operands (S / dX, A1, A2), the weight ring, the
// biases, the REINFORCE weights, barriers.
__host__ __device__ __forceinline__ int chain_stage_bytes(int max_n) { return 64 * r16(max_n); }
int bwd_chain_smem_bytes(int D, int H1, int H2, int max_n, int ns) {
  const int u = r16(D) + r16(H1) + r16(H2);
  return 256 * u + ns * chain_stage_bytes(max_n) + 4 * u + 128 * 4 + 5 * (int)sizeof(Prod) + 16 * ns + 32;
}

__global__ void __launch_bounds__(BC_THREADS) bwd_chain_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
                                                               const ChainWs cw, int ns, int max_n, int tmem_cols,
                                                               const int8_t* __restrict__ spins,
                                                               const double* __restrict__ logZR,
                                                               const float* __restrict__ logq,
                                                               const double* __restrict__ stats) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int k = find_inst(li, blockIdx.x);
  const InstDev& I = inst[k];
  const MadeDev& md = I.made;
  const int D = md.D, nh = md.nh, H1 = md.H1, H2 = md.H2, Dp = r16(D);
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const long long b0 = (long long)(blockIdx.x - li.tile_begin[k]) * 128;
  const int nv = min(128, li.batch - (int)b0);
  const int n_prod = 2 * nh + 1;
  unsigned char* sX = smem;  // S, then dX
  unsigned char* sA1 = sX + 256 * Dp;
  unsigned char* sA2 = sA1 + 256 * r16(H1);
  unsigned char* ring = sA2 + 256 * r16(H2);
  const int sbytes = chain_stage_bytes(max_n);
  float* sb = reinterpret_cast<float*>(ring + ns * sbytes);  // biases: hidden layers, output
  float* sw = sb + (Dp + r16(H1) + r16(H2));
  Prod* prod = reinterpret_cast<Prod*>(sw + 128);
  uint64_t* full = reinterpret_cast<uint64_t*>(prod + 5);  // a stage's weights have landed
  uint64_t* done = full + ns;   // a stage's MMAs
  uint64_t* pdone = done + ns;  // a product's
  uint32_t* slot = reinterpret_cast<uint32_t*>(pdone + 1);
  const ChainTile g(D, H1, H2);
  uint16_t* gt = cw.base + cw.off[k] + (long long)(blockIdx.x - li.tile_begin[k]) * g.elems;
  const uint16_t* tiles = md.ctiles;
  const int rp0 = nh >= 1 ? r16(H1) : Dp, rp1 = nh >= 2 ? r16(H2) : Dp;  // padded widths after layers 0, 1
  if (t == 0) {
    for (int i = 0; i < 2 * ns + 1; ++i) mbar_init(full + i, 1);
    // forward layers, then the transposed ones from the last down to the second
    for (int l = 0, off = 0; l <= nh; ++l) {
      const int rp = l == nh ? Dp : (l == 0 ? rp0 : rp1), cp = l == 0 ? Dp : (l == 1 ? rp0 : rp1);
      prod[l] = Prod{off, rp, cp, 0};
      if (l >= 1) prod[2 * nh + 1 - l] = Prod{off, rp, cp, 1};
      off += rp * cp;
    }
  }
  if (w == 0) {
    tc::tmem_alloc(slot, (uint32_t)tmem_cols);
    tc::tmem_relinquish();
  }
  {
    int so = 0;
    for (int l = 0; l <= nh; ++l) {
      const LayerDev& L = md.layer[l];
      const float* b = md.packed + L.dst_off + (long long)L.nout * L.nin;
      for (int n = t; n < r16(L.nout); n += BC_THREADS) sb[so + n] = n < L.nout ? __ldg(b + n) : 0.f;
      so += r16(L.nout);
    }
  }
  // the tile's spins: BF16 operand; 8 rows x 4 granules of 8 a warp (whole
  // sectors, conflict-free stores), one load a granule where aligned
  const int8_t* sp = spins + I.spin_units * li.batch + b0 * D;
  const bool al8 = (D & 7) == 0 && (reinterpret_cast<uintptr_t>(sp) & 7) == 0;
  for (int c0 = 0; c0 < (Dp >> 3); c0 += 4) {
    const int i0 = 8 * (c0 + (lane >> 3)), r = 8 * w + (t & 7);
    if (i0 >= Dp) continue;
    uint32_t lo = 0, hi = 0;  // the granule's spins, one byte each
    const int n8 = r < nv ? max(0, min(8, D - i0)) : 0;
    const int8_t* src = sp + (long long)r * D + i0;
    if (al8 && n8 == 8) {
      const uint2 q = __ldg(reinterpret_cast<const uint2*>(src));
      lo = q.x;
      hi = q.y;
    } else {
      for (int j = 0; j < n8; ++j) (j < 4 ? lo : hi) |= (uint32_t)(uint8_t)src[j] << (8 * (j & 3));
    }
    uint32_t h[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t v = 0;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int i = 2 * q + j;
        const int8_t s = (int8_t)((i < 4 ? lo : hi) >> (8 * (i & 3)));
        v |= (i < n8 ? (s > 0 ? 0x3F80u : 0xBF80u) : 0u) << (16 * j);
      }
      h[q] = v;
    }
    *reinterpret_cast<uint4*>(sX + k_off(r, i0, Dp)) = make_uint4(h[0], h[1], h[2], h[3]);
  }
  if (t < 128) {
    float wv = 0.f;
    if (t < nv) {
      const double sc = -1.0 / (li.beta[k] * stats_batch(stats + 8 * k));
      const long long o = (long long)k * li.batch + b0 + t;
      wv = (float)(sc * (logZR[o] - (double)logq[o] - stats[8 * k + 4]));
    }
    sw[t] = wv;
  }
  fence_proxy_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *slot;
  bool ok = true;
  // warp 0: weight stages fetched / used over all products, the next to fetch
  int issued = 0, used = 0, fp = 0, fs = 0;
  auto fetch_next = [&]() {
    if (fp == n_prod) return;
    fetch(prod[fp], fs, tiles, ring + (issued % ns) * sbytes, &full[issued % ns], lane);
    ++issued;
    if (++fs == (prod[fp].K() + 31) >> 5) ++fp, fs = 0;
  };
  if (w == 0)
    for (int i = 0; i < ns - 1; ++i) fetch_next();
  const int row = 32 * (w & 3) + lane;  // the TMEM lane this thread reads
  const uint32_t trow = tmem + ((uint32_t)(32 * (w & 3)) << 16);
  const float wrow = sw[row];
  const bool rowv = row < nv;
  int so = 0;  // the forward layer's biases
  for (int p = 0; p < n_prod; ++p) {
    const Prod P = prod[p];
    const int Np = P.N(), Kp = P.K();
    const bool tr = P.tr != 0;
    // A operand and the buffer the result goes to: 0 X / S, 1 A1, 2 A2
    const int src = tr ? (p == nh + 1 ? 0 : 2) : p;
    const int dst = tr ? 2 * nh + 1 - p : (p == nh ? 0 : p + 1);
    unsigned char* sA = src == 0 ? sX : (src == 1 ? sA1 : sA2);
    unsigned char* sO = dst == 0 ? sX : (dst == 1 ? sA1 : sA2);
    if (w == 0) {
      const int gsrc = !tr ? (src == 0 ? g.S : (src == 1 ? g.A1 : g.A2)) : (src == 0 ? g.X : g.dA2);
      if (lane == 0) bulk_s2g(gt + gsrc, sA, 256u * (uint32_t)Kp);  // the operand, finished before the last barrier
      const uint32_t id = tc::idesc(128, Np, 1u) | (tr ? 1u << 16 : 0u);
      const int nk = (Kp + 31) >> 5;
      for (int ks = 0; ks < nk && ok; ++ks) {
        const int st = used % ns;
        if (!mbar_wait(&full[st], (uint32_t)((used / ns) & 1))) {
          ok = false;
          break;
        }
        if (lane == 0) {
          const uint32_t b = smem_u32(ring + st * sbytes);
#pragma unroll
          for (int kk = 0; kk < 2; ++kk) {
            if (ks * 32 + kk * 16 >= Kp) break;
            const uint64_t da = tc::smem_desc(smem_u32(sA) + (uint32_t)(ks * 2 + kk) * 256u, 128u, (uint32_t)Kp * 16u);
            const uint64_t db = tr ? tc::smem_desc(b + (uint32_t)(kk * 32 * Np), 16u * (uint32_t)Np, 128u)
                                   : tc::smem_desc(b + kk * 256u, 128u, 512u);
            tc::mma_bf16(tmem, da, db, id, (ks > 0 || kk > 0) ? 1u : 0u);
          }
          tc::mma_commit(&done[st]);
        }
        __syncwarp();
        ++used;
        // the next fetch takes the slot of the stage before this one: its MMAs first
        if (used >= 2 && !mbar_wait(&done[(used - 2) % ns], (uint32_t)(((used - 2) / ns) & 1))) {
          ok = false;
          break;
        }
        fetch_next();
      }
      if (ok && lane == 0) {
        bulk_wait_read();  // the buffer written below has been copied out
        tc::mma_commit(pdone);
      }
      __syncwarp();
    }
    ok = mbar_wait(pdone, (uint32_t)(p & 1)) && ok;
    tc::fence_after_sync();
    if (ok) {
      for (int c = w >> 2; c < (Np >> 4); c += BC_THREADS / 128) {
        const int n0 = 16 * c;
        float v[16];
        tc::tmem_ld16(trow + (uint32_t)n0, v);
        uint4* o0 = reinterpret_cast<uint4*>(sO + k_off(row, n0, Np));
        uint4* o1 = reinterpret_cast<uint4*>(sO + k_off(row, n0 + 8, Np));
        if (tr || p == nh) {
          const uint4 m0 = *o0, m1 = *o1;
          const uint32_t m[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
          if (tr) {  // the layer's own values mask its delta
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              v[2 * j] = bf_lo(m[j]) > 0.f ? v[2 * j] : 0.f;
              v[2 * j + 1] = bf_hi(m[j]) > 0.f ? v[2 * j + 1] : 0.f;
            }
          } else {  // the spins (0 past D and the batch) are what dX replaces
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float x = v[j] + sb[so + n0 + j], s = (j & 1) ? bf_hi(m[j >> 1]) : bf_lo(m[j >> 1]);
              v[j] = wrow * s / (1.f + expf(s * x));
            }
          }
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = rowv ? fmaxf(v[j] + sb[so + n0 + j], 0.f) : 0.f;
        }
        *o0 = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
        *o1 = make_uint4(pack2(v[8], v[9]), pack2(v[10], v[11]), pack2(v[12], v[13]), pack2(v[14], v[15]));
      }
    }
    if (!tr) so += Np;
    // results visible to the next product's MMAs and copies, TMEM reads before its writes
    fence_proxy_async_smem();
    tc::fence_before_sync();
    ok = __syncthreads_and(ok) != 0;
    tc::fence_after_sync();
    if (!ok) break;
  }
  if (t == 0) {  // the last result
    if (ok) bulk_s2g(gt + (nh == 0 ? g.X : g.dA1), nh == 0 ? sX : sA1, 256u * (uint32_t)(nh == 0 ? Dp : r16(H1)));
    bulk_wait_read();
  }
  if (!ok) {
    // copies and MMAs still in flight get a bounded time to finish
    if (w == 0) {
      for (int i = max(0, issued - ns); i < issued; ++i) mbar_wait(&full[i % ns], (uint32_t)((i / ns) & 1));
      for (int i = max(0, used - ns); i < used; ++i) mbar_wait(&done[i % ns], (uint32_t)((i / ns) & 1));
    }
    if (t == 0) atomicExch(li.status, 2);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (w == 0) tc::tmem_dealloc(tmem, (uint32_t)tmem_cols);
}

// Weight gradients: dW_l = delta_l^T act_l over the samples, one CTA per 128
// rows of a weight matrix (all columns, at most 256) and slice of the batch.
// The chain's tiles are the operands as they stand: their core matrices hold 8
// samples x 8 units with the units contiguous, which is the MN-major operand
// of this product (K = samples), so a stage is 17 bulk copies (16 groups of 8
// samples of the CTA's rows, the other operand whole) into a two-slot ring and
// the threads touch no operand.  A constant tile with a column of ones gives
// the bias gradient in 16 columns of its own.  Bound by the copies (96 KB a
// 256 x 256 stage) and the epilogue.
#define BW_A_BYTES (16 * 2048)
__host__ __device__ __forceinline__ int chain_wgrad_smem(int max_n) {
  return 2 * (BW_A_BYTES + 256 * r16(max_n)) + 4096 + 64;
}
__global__ void __launch_bounds__(128) chain_wgrad_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
                                                          const ChainWs cw, int splits, int max_n, int tmem_cols,
                                                          float* __restrict__ partials, long long part_stride) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int k = find_inst(li, blockIdx.x);
  const MadeDev& md = inst[k].made;
  const int nh = md.nh, D = md.D;
  int l = 0, mb = blockIdx.x - li.tile_begin[k];
  for (; l < nh; ++l) {
    const int cnt = (md.layer[l].nout + 127) >> 7;
    if (mb < cnt) break;
    mb -= cnt;
  }
  const int M = md.layer[l].nout, N = md.layer[l].nin, Np = r16(N), Mp = r16(M), m0 = 128 * mb;
  const int mw = min(128, Mp - m0);
  const ChainTile g(D, md.H1, md.H2);
  const uint16_t* A = cw.base + cw.off[k] + (l == nh ? g.X : (l == 1 ? g.dA2 : g.dA1));
  const uint16_t* B = cw.base + cw.off[k] + (l == 0 ? g.S : (l == 1 ? g.A1 : g.A2));
  const int ntile = (li.batch + 127) / 128, per = (ntile + splits - 1) / splits;
  const int t_lo = blockIdx.y * per, nt = max(0, min(ntile, t_lo + per) - t_lo);
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const int sbytes = BW_A_BYTES + 256 * r16(max_n);
  unsigned char* ones = smem + 2 * sbytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(ones + 4096);  // [2] operands landed
  uint64_t* mma = full + 2;                                   // [2] stage's products done
  uint64_t* done = mma + 2;
  uint32_t* slot = reinterpret_cast<uint32_t*>(done + 1);
  if (t == 0)
    for (int i = 0; i < 5; ++i) mbar_init(full + i, 1);
  if (w == 0) {
    tc::tmem_alloc(slot, (uint32_t)tmem_cols);
    tc::tmem_relinquish();
  }
  // ones[k][n]: 16 columns, the first 1
  for (int e = t; e < 256; e += 128) {  // 16-byte rows: sample e >> 1, columns 8 (e & 1) ..
    const int s = e >> 1, c = e & 1;
    *reinterpret_cast<uint4*>(ones + (s >> 3) * 256 + c * 128 + (s & 7) * 16) = make_uint4(c ? 0u : 0x3F80u, 0, 0, 0);
  }
  fence_proxy_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *slot;
  bool ok = true;
  if (w == 0) {
    auto load = [&](int i) {
      unsigned char* s = smem + (i & 1) * sbytes;
      const long long o = (long long)(t_lo + i) * g.elems;
      if (lane == 0) mbar_expect_tx(&full[i & 1], 16u * 16u * (uint32_t)mw + 256u * (uint32_t)Np);
      __syncwarp();
      if (lane < 16) bulk_g2s(s + 2048 * lane, A + o + (long long)lane * 8 * Mp + 8 * m0, 16u * (uint32_t)mw, &full[i & 1]);
      else if (lane == 16) bulk_g2s(s + BW_A_BYTES, B + o, 256u * (uint32_t)Np, &full[i & 1]);
    };
    const uint32_t id = tc::idesc(128, Np, 1u) | (1u << 15) | (1u << 16);
    const uint32_t id1 = tc::idesc(128, 16, 1u) | (1u << 15) | (1u << 16);
    if (nt > 0) load(0);
    if (nt > 1) load(1);
    int issued = min(nt, 2);
    for (int i = 0; i < nt; ++i) {
      if (!mbar_wait(&full[i & 1], (uint32_t)((i >> 1) & 1))) {
        ok = false;
        break;
      }
      if (lane == 0) {
        const uint32_t a = smem_u32(smem + (i & 1) * sbytes), b = a + BW_A_BYTES;
        for (int kk = 0; kk < 8; ++kk) {  // 16 samples each
          const uint64_t da = tc::smem_desc(a + (uint32_t)kk * 4096u, 2048u, 128u);
          tc::mma_bf16(tmem, da, tc::smem_desc(b + (uint32_t)kk * 32u * (uint32_t)Np, 16u * (uint32_t)Np, 128u), id,
                       (i > 0 || kk > 0) ? 1u : 0u);
          tc::mma_bf16(tmem + (uint32_t)Np, da, tc::smem_desc(smem_u32(ones) + (uint32_t)kk * 512u, 256u, 128u), id1,
                       (i > 0 || kk > 0) ? 1u : 0u);
        }
        tc::mma_commit(&mma[i & 1]);
        if (i == nt - 1) tc::mma_commit(done);
      }
      __syncwarp();
      if (i >= 1 && i + 1 < nt) {  // the slot of tile i - 1 takes tile i + 1
        if (!mbar_wait(&mma[(i - 1) & 1], (uint32_t)(((i - 1) >> 1) & 1))) {
          ok = false;
          break;
        }
        load(i + 1);
        ++issued;
      }
    }
    if (!ok)  // copies still in flight get a bounded time to land
      for (int i = max(0, issued - 2); i < issued; ++i) mbar_wait(&full[i & 1], (uint32_t)((i >> 1) & 1));
  }
  if (nt > 0) ok = mbar_wait(done, 0) && ok;
  ok = __syncthreads_and(ok) != 0;
  tc::fence_after_sync();
  if (ok) {
    // 32 x 32 blocks through shared memory (the stages are free), so that rows go out whole
    float* G = partials + ((long long)k * splits + blockIdx.y) * part_stride + md.layer[l].dst_off;
    float* stg = reinterpret_cast<float*>(smem) + w * 32 * 33;
    const uint32_t tw = tmem + ((uint32_t)(32 * w) << 16);
    const int mr = m0 + 32 * w;
    for (int c0 = 0; c0 < Np; c0 += 32) {
      float v[2][16];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (nt > 0 && c0 + 16 * h < Np) tc::tmem_ld16(tw + (uint32_t)(c0 + 16 * h), v[h]);
        else
#pragma unroll
          for (int j = 0; j < 16; ++j) v[h][j] = 0.f;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int j = 0; j < 16; ++j) stg[lane * 33 + 16 * h + j] = v[h][j];
      __syncwarp();
      if (c0 + lane < N)
#pragma unroll 8
        for (int r = 0; r < 32; ++r)
          if (mr + r < M) G[(long long)(mr + r) * N + c0 + lane] = stg[r * 33 + lane];
      __syncwarp();
    }
    float v[16];
    if (nt > 0) tc::tmem_ld16(tw + (uint32_t)Np, v);
    else v[0] = 0.f;
    if (mr + lane < M) G[(long long)M * N + mr + lane] = v[0];
  } else if (t == 0) {
    atomicExch(li.status, 2);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (w == 0) tc::tmem_dealloc(tmem, (uint32_t)tmem_cols);
}

int chain_wgrad_smem_bytes(int max_n) { return chain_wgrad_smem(max_n); }

cudaError_t launch_chain_wgrad(const InstDev* d_inst, const LaunchInfo& li, const ChainWs& cw, int splits, int max_n,
                               float* partials, long long part_stride, cudaStream_t s) {
  const int nblk = li.tile_begin[li.n_inst];
  if (nblk == 0) return cudaSuccess;
  int cols = 32;
  while (cols < r16(max_n) + 16) cols *= 2;
  const int smem = chain_wgrad_smem(max_n);
  cudaError_t e = cudaFuncSetAttribute(chain_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  chain_wgrad_kernel<<<dim3(nblk, splits), 128, smem, s>>>(d_inst, li, cw, splits, max_n, cols, partials, part_stride);
  return cudaGetLastError();
}

cudaError_t launch_bwd_chain(const InstDev* d_inst, const LaunchInfo& li, const ChainWs& cw, int ns, int max_n,
                             int smem_bytes, const int8_t* spins, const double* logZR, const float* logq,
                             const double* stats, cudaStream_t s) {
  const int nblk = li.tile_begin[li.n_inst];
  if (nblk == 0) return cudaSuccess;
  int cols = 32;
  while (cols < r16(max_n)) cols *= 2;
  cudaError_t e = cudaFuncSetAttribute(bwd_chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  bwd_chain_kernel<<<nblk, BC_THREADS, smem_bytes, s>>>(d_inst, li, cw, ns, max_n, cols, spins, logZR, logq, stats);
  return cudaGetLastError();
}

}  // namespace tnvan
