// Hidden values, dX and deltas of the BF16 REINFORCE backward (Eq. 10) on
// tcgen05, for networks the fused kernel (k_bwd_fused.cu) does not take: up to
// two hidden layers and D of at most 256 units each.
//
// One CTA (256 threads) takes 128 samples through every layer:
//   A1 = relu(S W1^T + b1), A2 = relu(A1 W2^T + b2),
//   dX = w s sigmoid(-s (A2 Wo^T + bo)),
//   dA2 = (dX Wo) 1[A2 > 0], dA1 = (dA2 W2) 1[A1 > 0],
// each rounded to BF16 as the next product's operand and kept in shared memory
// (K-major core matrices; dX takes S's place, dA2 A2's and dA1 A1's), with one
// row-major BF16 copy of each and of S in global memory for the weight
// gradients (k_gemm.cu).  Weights come from the packed BF16 network through a
// ring of 32-input stages, the next product's first stages fetched before this
// product's epilogue; accumulators in TMEM, K in steps of 16 in input order.
// Bound by latency: five dependent products of 1 to 8 stages, each with an
// epilogue of (columns / 2) values a thread.  As five GEMM launches (64 columns
// a CTA, operands through global memory) with the weights' and spins' own
// launch before them, 134 us for the 48-256-256-48 network and 3 x 4,096
// samples; 73 us in this form.
#include <cuda_bf16.h>

#include "common.cuh"
#include "tc.cuh"

namespace tnvan {

#define BC_K 32                                // inputs per weight stage
#define BC_MN_SBO (BC_K * 2 / 16 * 128 + 16)  // 8-unit group stride of a transposed (MN-major) stage

namespace {

__device__ __forceinline__ void cp16(unsigned char* dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(src_bytes)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__host__ __device__ __forceinline__ int r16(int n) { return (n + 15) & ~15; }
__host__ __device__ __forceinline__ int r8(int n) { return (n + 7) & ~7; }

// Byte offset of element (row r, column k) of a K-major operand of kp columns.
__device__ __forceinline__ uint32_t k_off(int r, int k, int kp) { return tc::kmajor_off(r, k, kp * 2, 2); }

enum { BC_RELU, BC_DX, BC_MASK };

// One product of the chain: out [128 x N] from the operand A [128 x K] in
// shared memory (Kp columns) and the weights W [rows][cols] (BF16, row-major):
// forward N = rows, K = cols; transposed N = cols, K = rows.
struct Prod {
  const uint16_t* W;
  int rows, cols;
  bool tr;
  __device__ int N() const { return tr ? cols : rows; }
  __device__ int K() const { return tr ? rows : cols; }
  __device__ int stages() const { return (K() + BC_K - 1) / BC_K; }
};

// Stage ks of a product's weights into dst: forward K-major [N][32], transposed
// MN-major; zeros outside W.  16-byte asynchronous copies where the rows are
// aligned, else element by element.
__device__ void fetch(const Prod& p, int ks, unsigned char* dst, int t) {
  const int np = r16(p.N()), k0 = ks * BC_K;
  const bool al = (p.cols & 7) == 0 && (reinterpret_cast<uintptr_t>(p.W) & 15) == 0;
  if (!p.tr) {
    for (int u = t; u < np * (BC_K / 8); u += 256) {
      const int r = u >> 2, kq = (u & 3) * 8, gk = k0 + kq;
      unsigned char* d = dst + tc::kmajor_off(r, kq, BC_K * 2, 2);
      const int nv = r < p.rows ? max(0, min(8, p.cols - gk)) : 0;
      const uint16_t* src = p.W + (long long)r * p.cols + gk;
      if (al) {
        cp16(d, nv ? src : p.W, 2u * (uint32_t)nv);
      } else {
        uint32_t h[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          h[j] = (uint32_t)(2 * j < nv ? src[2 * j] : 0) | ((uint32_t)(2 * j + 1 < nv ? src[2 * j + 1] : 0) << 16);
        *reinterpret_cast<uint4*>(d) = make_uint4(h[0], h[1], h[2], h[3]);
      }
    }
  } else {
    const int rg = np >> 3;
    for (int u = t; u < rg * BC_K; u += 256) {
      const int k = u / rg, n = (u - k * rg) * 8, gk = k0 + k;
      unsigned char* d = dst + (n >> 3) * BC_MN_SBO + (k >> 3) * 128 + (k & 7) * 16;
      const int nv = gk < p.rows ? max(0, min(8, p.cols - n)) : 0;
      const uint16_t* src = p.W + (long long)gk * p.cols + n;
      if (al) {
        cp16(d, nv ? src : p.W, 2u * (uint32_t)nv);
      } else {
        uint32_t h[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          h[j] = (uint32_t)(2 * j < nv ? src[2 * j] : 0) | ((uint32_t)(2 * j + 1 < nv ? src[2 * j + 1] : 0) << 16);
        *reinterpret_cast<uint4*>(d) = make_uint4(h[0], h[1], h[2], h[3]);
      }
    }
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
// REINFORCE weights, barriers.
__host__ __device__ __forceinline__ int chain_stage_bytes(int max_n) { return r16(max_n) / 8 * BC_MN_SBO; }
int bwd_chain_smem_bytes(int D, int H1, int H2, int max_n, int ns) {
  return 128 * 2 * (r16(D) + r16(H1) + r16(H2)) + ns * chain_stage_bytes(max_n) + 128 * 4 + 8 * ns + 16;
}

__global__ void __launch_bounds__(256) bwd_chain_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
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
  const int t = threadIdx.x, w = t >> 5;
  const long long b0 = (long long)(blockIdx.x - li.tile_begin[k]) * 128;
  const int nv = min(128, li.batch - (int)b0);
  unsigned char* sX = smem;  // S, then dX
  unsigned char* sA1 = sX + 256 * Dp;
  unsigned char* sA2 = sA1 + 256 * r16(H1);
  unsigned char* ring = sA2 + 256 * r16(H2);
  const int sbytes = chain_stage_bytes(max_n);
  float* sw = reinterpret_cast<float*>(ring + ns * sbytes);
  uint64_t* bar = reinterpret_cast<uint64_t*>(sw + 128);
  uint32_t* slot = reinterpret_cast<uint32_t*>(bar + ns);
  const ChainRows g = chain_rows(cw, k, li.batch, D, H1, H2);
  // the products in order
  const LayerDev* L = md.layer;
  Prod prod[5];
  int epi[5], n_prod = 0;
  for (int l = 0; l < nh; ++l) {
    prod[n_prod] = Prod{md.packed16 + L[l].dst_off, L[l].nout, L[l].nin, false};
    epi[n_prod++] = BC_RELU;
  }
  prod[n_prod] = Prod{md.packed16 + L[nh].dst_off, L[nh].nout, L[nh].nin, false};
  epi[n_prod++] = BC_DX;
  for (int l = nh; l >= 1; --l) {
    prod[n_prod] = Prod{md.packed16 + L[l].dst_off, L[l].nout, L[l].nin, true};
    epi[n_prod++] = BC_MASK;
  }
  if (t == 0)
    for (int i = 0; i < ns; ++i) mbar_init(&bar[i], 1);
  if (w == 0) {
    tc::tmem_alloc(slot, (uint32_t)tmem_cols);
    tc::tmem_relinquish();
  }
  int issued = 0, used = 0;  // weight stages fetched / used, over all products
  int fp = 0, fs = 0;        // the next stage to fetch
  auto fetch_next = [&]() {  // one copy group per call
    if (fp < n_prod) {
      fetch(prod[fp], fs, ring + (issued % ns) * sbytes, t);
      ++issued;
      if (++fs == prod[fp].stages()) ++fp, fs = 0;
    }
    cp_commit();
  };
  for (int i = 0; i < ns - 1; ++i) fetch_next();
  // the tile's spins: BF16 operand and global copy; 8 rows x 4 granules of 8 a
  // warp (whole sectors, conflict-free stores), one load a granule where aligned
  const int8_t* sp = spins + I.spin_units * li.batch + b0 * D;
  const bool al8 = (D & 7) == 0 && (reinterpret_cast<uintptr_t>(sp) & 7) == 0;
  for (int c0 = 0; c0 < (Dp >> 3); c0 += 4) {
    const int i0 = 8 * (c0 + ((t >> 3) & 3));
    if (i0 >= Dp) continue;
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      const int r = 64 * rr + 8 * w + (t & 7);
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
      const uint4 u = make_uint4(h[0], h[1], h[2], h[3]);
      *reinterpret_cast<uint4*>(sX + k_off(r, i0, Dp)) = u;
      if (r < nv && i0 < g.ldD) *reinterpret_cast<uint4*>(g.S + (b0 + r) * g.ldD + i0) = u;
    }
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
  const int row = 32 * (w & 3) + (t & 31);  // the TMEM lane this thread reads
  const long long grow = b0 + row;
  for (int p = 0; p < n_prod && ok; ++p) {
    const int N = prod[p].N(), Np = r16(N), K = prod[p].K(), Kp = r16(K), nk = prod[p].stages();
    const bool tr = prod[p].tr;
    // A operand and the buffer the result goes to
    const int src = tr ? (p == nh + 1 ? 0 : 2) : p;       // 0: X / S, 1: A1, 2: A2
    const int dst = tr ? 2 * nh + 1 - p : (p == nh ? 0 : p + 1);
    const unsigned char* sA = src == 0 ? sX : (src == 1 ? sA1 : sA2);
    unsigned char* sO = dst == 0 ? sX : (dst == 1 ? sA1 : sA2);
    const uint32_t id = tc::idesc(128, Np, 1u) | (tr ? 1u << 16 : 0u);
    for (int ks = 0; ks < nk; ++ks) {
      const int st = used % ns;
      if (ns == 2) cp_wait<0>();
      else if (ns == 3) cp_wait<1>();
      else cp_wait<2>();
      fence_proxy_async_smem();
      tc::fence_before_sync();
      __syncthreads();
      tc::fence_after_sync();
      if (t == 0) {
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
          if (ks * BC_K + kk * 16 >= Kp) break;
          const uint64_t a = tc::smem_desc(smem_u32(sA) + (uint32_t)(ks * 2 + kk) * 256u, 128u, (uint32_t)Kp * 16u);
          const uint64_t b = tc::smem_desc(smem_u32(ring + st * sbytes) + kk * 256u, 128u,
                                           tr ? BC_MN_SBO : BC_K * 2 / 16 * 128);
          tc::mma_bf16(tmem, a, b, id, (ks > 0 || kk > 0) ? 1u : 0u);
        }
        tc::mma_commit(&bar[st]);
      }
      // the next fetch reuses the slot of stage used - 1: its MMAs first
      if (used >= 1 && !mbar_wait(&bar[(used - 1) % ns], (uint32_t)(((used - 1) / ns) & 1))) ok = false;
      ++used;
      if (ok) fetch_next();
      else cp_commit();
    }
    if (ok && !mbar_wait(&bar[(used - 1) % ns], (uint32_t)(((used - 1) / ns) & 1))) ok = false;
    tc::fence_after_sync();
    ok = __syncthreads_and(ok) != 0;
    if (!ok) break;
    // epilogue: row `row`, half of the columns per warpgroup
    const float* bias = tr ? nullptr : md.packed + L[p].dst_off + (long long)L[p].nout * L[p].nin;
    uint16_t* gout = p < nh ? (p == 0 ? g.A1 : g.A2) : (p == nh ? g.X : (dst == 2 ? g.dA2 : g.dA1));
    const int ld = dst == 0 ? g.ldD : (dst == 1 ? g.ld1 : g.ld2);
    const float wrow = sw[row];
    const bool rowv = row < nv;
    const int nc = Np >> 4, c_lo = (w >> 2) ? (nc + 1) >> 1 : 0, c_hi = (w >> 2) ? nc : (nc + 1) >> 1;
    for (int c = c_lo; c < c_hi; ++c) {
      float v[16];
      tc::tmem_ld16(tmem + ((uint32_t)(32 * (w & 3)) << 16) + 16u * (uint32_t)c, v);
      const int n0 = 16 * c;
      uint4* o0 = reinterpret_cast<uint4*>(sO + k_off(row, n0, Np));
      uint4* o1 = reinterpret_cast<uint4*>(sO + k_off(row, n0 + 8, Np));
      float r[16];
      if (epi[p] == BC_MASK) {
        const uint4 m0 = *o0, m1 = *o1;
        const uint32_t m[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          r[2 * j] = bf_lo(m[j]) > 0.f ? v[2 * j] : 0.f;
          r[2 * j + 1] = bf_hi(m[j]) > 0.f ? v[2 * j + 1] : 0.f;
        }
      } else if (epi[p] == BC_RELU) {
#pragma unroll
        for (int j = 0; j < 16; ++j) r[j] = n0 + j < N ? fmaxf(v[j] + __ldg(bias + n0 + j), 0.f) : 0.f;
      } else {  // the spins are what dX replaces
        const uint4 m0 = *o0, m1 = *o1;
        const uint32_t m[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          r[j] = 0.f;
          if (n0 + j < N && rowv) {
            const float x = v[j] + __ldg(bias + n0 + j), s = (j & 1) ? bf_hi(m[j >> 1]) : bf_lo(m[j >> 1]);
            r[j] = wrow * s / (1.f + expf(s * x));
          }
        }
      }
      const uint4 u0 = make_uint4(pack2(r[0], r[1]), pack2(r[2], r[3]), pack2(r[4], r[5]), pack2(r[6], r[7]));
      const uint4 u1 = make_uint4(pack2(r[8], r[9]), pack2(r[10], r[11]), pack2(r[12], r[13]), pack2(r[14], r[15]));
      *o0 = u0;
      *o1 = u1;
      if (rowv) {
        if (n0 < ld) *reinterpret_cast<uint4*>(gout + grow * ld + n0) = u0;
        if (n0 + 8 < ld) *reinterpret_cast<uint4*>(gout + grow * ld + n0 + 8) = u1;
      }
    }
    // results visible to the next product's MMAs (its first stage's barrier), TMEM reads before its writes
    fence_proxy_async_smem();
    tc::fence_before_sync();
  }
  cp_wait<0>();
  if (!ok) {
    // give the MMAs still in flight a bounded time to finish before TMEM is freed
    for (int i = 0; i < ns && i < used; ++i) mbar_wait(&bar[(used - 1 - i) % ns], (uint32_t)(((used - 1 - i) / ns) & 1));
    if (t == 0) atomicExch(li.status, 2);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (w == 0) tc::tmem_dealloc(tmem, (uint32_t)tmem_cols);
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
  bwd_chain_kernel<<<nblk, 256, smem_bytes, s>>>(d_inst, li, cw, ns, max_n, cols, spins, logZR, logq, stats);
  return cudaGetLastError();
}

}  // namespace tnvan
