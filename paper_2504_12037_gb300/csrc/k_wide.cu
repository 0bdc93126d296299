// Wide lattice strips: exact row transfer-matrix contraction (Eq. 2-4 with W
// = whole columns) of strips of up to TNVAN_WIDE_MAX_W columns, for lattice
// instances whose plan is an elimination plan (their strips are wider than
// the per-thread strip kernels hold in registers).  Forward log Z_R only.
//
// One warp per (sample, strip), four samples of one strip per CTA.  Per row y
// (same gauge as the strip planner: every vertical coupling >= 0):
//   v <- V_{y-1} v   with V the Kronecker product of [[1, t_c], [t_c, 1]],
//                    t_c = exp(-2 beta Jv_c);
//   v <- D_y v       D_y(x) = product over the row's bonds that x leaves
//                    unsatisfied (J s s' < 0, W neighbours included) of
//                    exp(-2 beta |J|): every factor is at most 1;
//   v <- v 2^k       where the row's largest entry has left [2^20, 2^81).
// ln Z_strip = ln sum_x v(x) - ln 2 sum k + beta sum |J| over the strip's
// bonds; log Z_R adds beta sum over W-W bonds J s s' (Eq. 4).
//
// The 2^w states of a row are spread over the warp: bits 0-4 of a state on the
// lane, the others on the register index j.  A vertical factor on a register
// bit is a pair of FMAs, on a lane bit a shuffle and an FMA per state.  Strips
// of 10 to 12 columns instead exchange the lane bits with register bits 0-4
// (32 x 32 transposes through shared memory), apply the five factors in
// registers and exchange back: four shared accesses per state, not five
// shuffles, without their latency chain.
// D_y of a state is a product over the bonds in column order, the W neighbours
// after bond 3 and last.  Its lane part is formed once per lane and row; the
// register part along the binary tree of j's bits, so a state costs about
// three products and not a chain of nine conditional ones.  Entries 2^-149 times
// the largest have to survive a row (at low temperature a frustrated row can
// make the next row's largest of them), so scales go into v, not into D, and
// before the largest entry falls below 1; keeping it near 2^50 leaves most rows
// without a scaling pass.  The factors are tabulated per strip row and beta
// (wide_tab_kernel).  Every value is rounded as in the
// plain chain of products: at high temperature the same few products recur in
// every row, so their rounding is systematic and moves log Z.
// Bound by the FP32 pipe and shared memory alike (w + 4 operations and 4
// shared accesses a state and row); 40 x 40 ferromagnet, 6 x 1,000 samples:
// 5.15 ms with conditional products per state, a sample per CTA and shuffles,
// 2.14 ms in this form (2.12 with the scales on the next row's diagonal, which
// lost the small entries, 2.24 with a scaling pass for every row below 1).
#include "common.cuh"

namespace tnvan {

namespace {

// Factor of a bond of coupling J that a state leaves unsatisfied.
__device__ __forceinline__ float unsat_factor(float J, float beta) { return expf(-2.f * beta * fabsf(J)); }

// Per strip row 32 floats: 0-10 the horizontal bonds' factors, 16-27 the
// vertical factors from the row above, 28 the mask of negative horizontal
// couplings as bits, 30 / 31 the W neighbours' factors.
constexpr int ROW_FLOATS = 32;

}  // namespace

// States per lane of a strip of w columns.
__host__ __device__ __forceinline__ int wide_npl(int w) { return w <= 5 ? 1 : 1 << (w - 5); }

int wide_tab_floats(int L) { return L * ROW_FLOATS; }

// One warp per strip row of an instance.
__global__ void __launch_bounds__(128) wide_tab_kernel(const InstDev* __restrict__ inst, const LaunchInfo li) {
  const int k = blockIdx.y;
  if (li.tile_begin[k + 1] == li.tile_begin[k]) return;
  const InstDev& I = inst[k];
  int st = 0, y = blockIdx.x * 4 + (threadIdx.x >> 5);
  for (; st < I.n_wide; ++st) {
    if (y < I.wide[st].L) break;
    y -= I.wide[st].L;
  }
  if (st == I.n_wide) return;
  const WideRow* rows = I.wrows + I.wide[st].row0;
  const WideRow& R = rows[y];
  const int w = I.wide[st].w, t = threadIdx.x & 31;
  const float beta = (float)li.beta[k];
  float v = 1.f;
  if (t < w - 1) {
    v = unsat_factor(R.Jh[t], beta);
  } else if (t >= 16 && t < 16 + w && y > 0) {
    v = expf(-2.f * beta * rows[y - 1].Jv[t - 16]);
  } else if (t == 28) {
    uint32_t neg = 0;
    for (int c = 0; c + 1 < w; ++c) neg |= (R.Jh[c] < 0.f ? 1u : 0u) << c;
    v = __uint_as_float(neg);
  } else if (t == 30 && R.posL >= 0) {
    v = unsat_factor(R.JL, beta);
  } else if (t == 31 && R.posR >= 0) {
    v = unsat_factor(R.JR, beta);
  }
  I.wtab[I.wide[st].tab_off + y * ROW_FLOATS + t] = v;
}

namespace {

// v <- (I + t X_bit) v on register bit Q.
template <int NPL, int Q>
__device__ __forceinline__ void vert(float (&v)[NPL], float t) {
  if constexpr ((1 << Q) < NPL) {
#pragma unroll
    for (int j = 0; j < NPL; ++j) {
      if ((j >> Q) & 1) continue;
      const float a = v[j], b = v[j | (1 << Q)];
      v[j] = fmaf(t, b, a);
      v[j | (1 << Q)] = fmaf(t, a, b);
    }
  }
}

// The factors t[0..4] of the lane bits: 32 registers at a time exchanged with
// the lanes (two alternating shared buffers of 32 x 33 floats), applied as
// register bits, exchanged back.
template <int NPL>
__device__ __forceinline__ void vert_lanes(float (&v)[NPL], const float (&t)[5], float* buf, int lane) {
#pragma unroll
  for (int h = 0; h < NPL / 32; ++h) {
    float* b = buf + (h & 1) * (32 * 33);
    float x[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) b[j * 33 + lane] = v[h * 32 + j];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 32; ++j) x[j] = b[lane * 33 + j];
    vert<32, 0>(x, t[0]);
    vert<32, 1>(x, t[1]);
    vert<32, 2>(x, t[2]);
    vert<32, 3>(x, t[3]);
    vert<32, 4>(x, t[4]);
#pragma unroll
    for (int j = 0; j < 32; ++j) b[lane * 33 + j] = x[j];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 32; ++j) v[h * 32 + j] = b[j * 33 + lane];
  }
}

// The row's largest entry over the warp -> its exponent.
template <int NPL>
__device__ __forceinline__ int row_exponent(const float (&v)[NPL]) {
  float mx = 0.f;
#pragma unroll
  for (int j = 0; j < NPL; ++j) mx = fmaxf(mx, v[j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  return exponent_of(mx);
}

// Brings the largest entry, of exponent e, back to 2^50 where it has left the
// range; e2 counts the powers of two taken out.
#define WIDE_EXP 50
template <int NPL>
__device__ __forceinline__ void rescale(float (&v)[NPL], int& e, int& e2) {
  if (e >= WIDE_EXP - 30 && e <= WIDE_EXP + 30) return;  // the same for the warp
  const int k = min(WIDE_EXP - e, 127);  // no entry left: any
  const float sc = pow2i(k);
#pragma unroll
  for (int j = 0; j < NPL; ++j) v[j] *= sc;
  e += k;
  e2 -= k;
}

// Which lane bits a bond of the lane part leaves unsatisfied: bits i, i + 1.
__device__ __forceinline__ bool unsat(uint32_t x, int i, uint32_t neg_bit) {
  return (((x >> i) ^ (x >> (i + 1))) & 1u) != (neg_bit & 1u);
}

// The register part of D: p the product so far at the low LEV bits J of the
// register index; f[i][1 or 0] the factor of bond 5 + i when register bits i
// and i + 1 differ or agree, g the right neighbour's by the top bit.
template <int NPL, int LEV, int J, bool FIRST>
__device__ __forceinline__ void diag_tree(float (&v)[NPL], float p, const float (&f)[6][2], const float (&g)[2]) {
  if constexpr ((1 << LEV) == NPL) {
    const float d = p * g[(J >> (LEV - 1)) & 1];
    v[J] = FIRST ? d : v[J] * d;
  } else {
    constexpr int top = (J >> (LEV - 1)) & 1;
    diag_tree<NPL, LEV + 1, J, FIRST>(v, p * f[LEV - 1][top], f, g);
    diag_tree<NPL, LEV + 1, J | (1 << LEV), FIRST>(v, p * f[LEV - 1][top ^ 1], f, g);
  }
}

// D of a row on v (FIRST: v = 2^WIDE_EXP D).
template <int NPL, bool FIRST>
__device__ __forceinline__ void diag(float (&v)[NPL], const float* __restrict__ row, int w, uint32_t wantL,
                                     uint32_t wantR, bool hasL, bool hasR, int lane) {
  const float4 u03 = __ldg(reinterpret_cast<const float4*>(row));
  const float u[4] = {u03.x, u03.y, u03.z, u03.w};
  const uint32_t neg = __float_as_uint(__ldg(row + 28)), x0 = (uint32_t)lane;
  float pl = FIRST ? pow2i(WIDE_EXP) : 1.f;
#pragma unroll
  for (int c = 0; c < 4; ++c)
    if (c + 1 < w && unsat(x0, c, neg >> c)) pl *= u[c];
  if (hasL && (x0 & 1u) != wantL) pl *= __ldg(row + 30);
  if (w <= 5 && hasR && ((x0 >> (w - 1)) & 1u) != wantR) pl *= __ldg(row + 31);
  if constexpr (NPL == 1) {
    const float d = lane < (1 << w) ? pl : 0.f;
    v[0] = FIRST ? d : v[0] * d;
  } else {
    const float4 u47 = __ldg(reinterpret_cast<const float4*>(row + 4));
    const float4 u8 = __ldg(reinterpret_cast<const float4*>(row + 8));
    const float ub[6] = {u47.y, u47.z, u47.w, u8.x, u8.y, u8.z};
    float f[6][2];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const bool ng = (neg >> (5 + i)) & 1u;
      f[i][0] = ng ? ub[i] : 1.f;
      f[i][1] = ng ? 1.f : ub[i];
    }
    const float uR = hasR ? __ldg(row + 31) : 1.f;
    const float g[2] = {wantR ? uR : 1.f, wantR ? 1.f : uR};
    // bond 4 joins lane bit 4 and register bit 0
    const bool one4 = ((x0 >> 4) & 1u) != ((neg >> 4) & 1u);  // register bit 0 that satisfies it
    diag_tree<NPL, 1, 0, FIRST>(v, one4 ? pl * u47.x : pl, f, g);
    diag_tree<NPL, 1, 1, FIRST>(v, one4 ? pl : pl * u47.x, f, g);
  }
}

// One strip for one sample; NPL = states per lane (2^(w-5), or 1 for w <= 5).
// Returns ln of the normalised sum and the power-of-two exponent count.
template <int NPL>
__device__ __forceinline__ void wide_chain(const WideStripDev& sd, const WideRow* __restrict__ rows,
                                           const float* __restrict__ tab, const int8_t* __restrict__ srow, float* buf,
                                           int lane, float& lnz, int& e2) {
  const int w = sd.w;
  float v[NPL];
  // the W neighbours of 32 rows at a time, one row per lane: bit y & 31 of
  // wl / wr = the bit value of column 0 / w - 1 that satisfies the bond
  uint32_t wl = 0, wr = 0, hl = 0, hr = 0;
  auto neighbours = [&](int y0) {
    const int y = y0 + lane;
    const bool on = y < sd.L;
    const int pL = on ? rows[y].posL : -1, pR = on ? rows[y].posR : -1;
    const float sL = pL >= 0 ? (float)srow[pL] : 0.f, sR = pR >= 0 ? (float)srow[pR] : 0.f;
    wl = __ballot_sync(0xffffffffu, on && rows[y].JL * sL < 0.f);
    wr = __ballot_sync(0xffffffffu, on && rows[y].JR * sR < 0.f);
    hl = __ballot_sync(0xffffffffu, pL >= 0);
    hr = __ballot_sync(0xffffffffu, pR >= 0);
  };
  neighbours(0);
  diag<NPL, true>(v, tab, w, wl & 1u, wr & 1u, hl & 1u, hr & 1u, lane);
  int e = row_exponent(v);
  e2 = -WIDE_EXP;
  rescale(v, e, e2);
  for (int y = 1; y < sd.L; ++y) {
    if ((y & 31) == 0) neighbours(y);
    const uint32_t b = 1u << (y & 31);
    const float* row = tab + y * ROW_FLOATS;
    const float4 ta = __ldg(reinterpret_cast<const float4*>(row + 16)), tb = __ldg(reinterpret_cast<const float4*>(row + 20)),
                 tc = __ldg(reinterpret_cast<const float4*>(row + 24));
    const float t5[5] = {ta.x, ta.y, ta.z, ta.w, tb.x};
    if constexpr (NPL >= 32) {
      vert_lanes(v, t5, buf, lane);
    } else {
#pragma unroll
      for (int c = 0; c < 5; ++c)
        if (c < w) {
#pragma unroll
          for (int j = 0; j < NPL; ++j) v[j] = fmaf(t5[c], __shfl_xor_sync(0xffffffffu, v[j], 1 << c), v[j]);
        }
    }
    vert<NPL, 0>(v, tb.y);
    vert<NPL, 1>(v, tb.z);
    vert<NPL, 2>(v, tb.w);
    vert<NPL, 3>(v, tc.x);
    vert<NPL, 4>(v, tc.y);
    vert<NPL, 5>(v, tc.z);
    vert<NPL, 6>(v, tc.w);
    diag<NPL, false>(v, row, w, (wl & b) ? 1u : 0u, (wr & b) ? 1u : 0u, hl & b, hr & b, lane);
    e = row_exponent(v);
    rescale(v, e, e2);
  }
  const float sc = pow2i(-e);
  e2 += e;
  float z = 0.f;
#pragma unroll
  for (int j = 0; j < NPL; ++j) z += v[j] * sc;
  z = warp_sum(z);
  lnz = logf(z);
}

}  // namespace

// The strips of one state-count class (wide_npl(w) == NPL): CTA = four
// samples of strip blockIdx.y of the class, a warp each; per-strip results to
// part[(k * batch + b) * li.tile_aux + strip].
template <int NPL>
__global__ void __launch_bounds__(128, NPL >= 128 ? 3 : 4)
    wide_kernel(const InstDev* __restrict__ inst, const LaunchInfo li, const int8_t* __restrict__ spins,
                double* __restrict__ part) {
  __shared__ float tr[NPL >= 32 ? 4 * 2 * 32 * 33 : 1];
  const int k = blockIdx.z;
  if (li.tile_begin[k + 1] == li.tile_begin[k]) return;
  const InstDev& I = inst[k];
  const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x * 4 + wp;
  int nth = blockIdx.y, st = 0;
  for (; st < I.n_wide; ++st)
    if (wide_npl(I.wide[st].w) == NPL && nth-- == 0) break;
  if (st == I.n_wide || b >= li.batch) return;
  const WideStripDev sd = I.wide[st];
  const int8_t* srow = spins + I.spin_units * li.batch + (long long)b * I.D;
  float lnz = 0.f;
  int e2 = 0;
  wide_chain<NPL>(sd, I.wrows + sd.row0, I.wtab + sd.tab_off, srow, tr + (NPL >= 32 ? wp * 2 * 32 * 33 : 0), lane, lnz,
                  e2);
  if (lane == 0)
    part[((long long)k * li.batch + b) * li.tile_aux + st] =
        (double)lnz + (double)e2 * 0.69314718055994530942 + li.beta[k] * sd.c_hat;
}

// log Z_R per sample: the strips' results in strip order plus the W-W term.
__global__ void wide_sum_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
                                const int8_t* __restrict__ spins, const double* __restrict__ part,
                                double* __restrict__ logZR) {
  const int k = blockIdx.y;
  const InstDev& I = inst[k];
  if (I.n_wide == 0 || li.tile_begin[k + 1] == li.tile_begin[k]) return;
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < li.batch; b += gridDim.x * blockDim.x) {
    const double* p = part + ((long long)k * li.batch + b) * li.tile_aux;
    double lz = 0.0;
    for (int st = 0; st < I.n_wide; ++st) lz += p[st];
    const int8_t* srow = spins + I.spin_units * li.batch + (long long)b * I.D;
    float e1 = 0.f;
    for (int e = 0; e < I.n_ww; ++e) {
      const EdgeWW q = I.ww[e];
      e1 = fmaf(q.J, (float)(srow[q.a] * srow[q.b]), e1);
    }
    logZR[(long long)k * li.batch + b] = lz + li.beta[k] * (double)e1;
  }
}

cudaError_t launch_wide(const InstDev* d_inst, const LaunchInfo& li, const int* strips_per_class, int max_strips,
                        int max_rows, const int8_t* spins, double* part, double* logZR, cudaStream_t s) {
  if (li.tile_begin[li.n_inst] == 0 || max_strips == 0) return cudaSuccess;
  LaunchInfo lw = li;
  lw.tile_aux = max_strips;
  wide_tab_kernel<<<dim3((unsigned)((max_rows + 3) / 4), li.n_inst), 128, 0, s>>>(d_inst, lw);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  for (int c = 7; c >= 0; --c) {  // the widest strips first
    const int n = strips_per_class[c];  // most strips of class c in one instance
    if (n == 0) continue;
    const dim3 grid((unsigned)((li.batch + 3) / 4), n, li.n_inst);
    switch (c) {
      case 0: wide_kernel<1><<<grid, 128, 0, s>>>(d_inst, lw, spins, part); break;
      case 1: wide_kernel<2><<<grid, 128, 0, s>>>(d_inst, lw, spins, part); break;
      case 2: wide_kernel<4><<<grid, 128, 0, s>>>(d_inst, lw, spins, part); break;
      case 3: wide_kernel<8><<<grid, 128, 0, s>>>(d_inst, lw, spins, part); break;
      case 4: wide_kernel<16><<<grid, 128, 0, s>>>(d_inst, lw, spins, part); break;
      case 5: wide_kernel<32><<<grid, 128, 0, s>>>(d_inst, lw, spins, part); break;
      case 6: wide_kernel<64><<<grid, 128, 0, s>>>(d_inst, lw, spins, part); break;
      default: wide_kernel<128><<<grid, 128, 0, s>>>(d_inst, lw, spins, part); break;
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  wide_sum_kernel<<<dim3((unsigned)((li.batch + 255) / 256), li.n_inst), 256, 0, s>>>(d_inst, lw, spins, part, logZR);
  return cudaGetLastError();
}

}  // namespace tnvan
