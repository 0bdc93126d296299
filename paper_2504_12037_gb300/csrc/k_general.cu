// General leftover components (e.g. random regular graphs): exact
// contraction of every connected component of R by variable elimination
// (Eq. 4), one program per component compiled by the host planner.
//
// Eliminating spin v multiplies every factor that contains v -- its field
// factor exp(beta h_v(s) r_v) from the width set, the Boltzmann matrices of its
// remaining bonds (Eq. 2) and the intermediate tables that contain it -- and
// sums v out, giving a table over its remaining neighbours (at most
// 2^TNVAN_MAX_ELIM_W entries).  The host compiles each step into a record and, per input table,
// an index map from the step's extended index (its out-scope spins and v) to
// the input's entry; the product of a step's bond factors depends only on
// that index and beta and is tabulated once per call (general_pp_kernel), so
// a table entry costs one field factor, one bond product and one load per
// input.  A group of lanes shares one sample and splits each table's entries;
// tables are laid out [entry][sample] per CTA (consecutive samples in
// consecutive words), in shared memory, or for large arenas in a per-CTA
// slice of global scratch.  Forward
// passes use reused offsets (a table's space is free once the step that
// consumes it has run); the reverse sweep keeps every table.  Every new table
// is renormalised by a power of two.  Factors are stored normalised (largest
// entry 1); the removed constants (beta |h_v| per field, beta |J| per bond)
// are added back in FP64.  With DB, every table entry carries its
// beta-derivative (forward mode).
#include <algorithm>
#include <climits>

#include "common.cuh"

namespace tnvan {

__device__ __forceinline__ int padded_bytes(int D) {
  int w4 = (D + 3) / 4;
  if ((w4 & 1) == 0) ++w4;
  return 4 * w4;
}

// One compiled elimination step (layout in GenDev).
struct StepRec {
  int m, fb, fc, nin, npair, ppo, mo, out_live, out_full;
  const int* io;  // n_in x (live offset, full offset, spins of the input)
  const int* pr;  // n_pair x (pair id, position of the neighbour in the out scope)
};

// What a sweep needs of a step: sizes, offsets (out and in[] live or full) and
// the sample's field on the eliminated spin; f the record's place in fprog.
struct Step {
  int m, nin, ppo, mo, out, in[3], f;
  float h;
};

__device__ __forceinline__ StepRec step_at(const GenDev& G, int g) {
  const int* F = G.fprog + G.fstep[g];
  StepRec r;
  r.m = F[0];
  r.fb = F[1];
  r.fc = F[2];
  r.nin = F[3];
  r.npair = F[4];
  r.ppo = F[5];
  r.mo = F[6];
  r.out_live = F[7];
  r.out_full = F[8];
  r.io = F + 9;
  r.pr = F + 9 + 3 * r.nin;
  return r;
}

// Width-set field on the eliminated spin: h = sum_w J_vw s_w.
__device__ __forceinline__ float field_of(const GenDev& G, int fb, int fc, const int8_t* s) {
  float h = 0.f;
  for (int f = fb; f < fb + fc; ++f) h = fmaf(G.fldJ[f], (float)s[G.fld[2 * f]], h);
  return h;
}

// The next GL steps of a sweep, one per lane of the group: their records and
// fields are chains of dependent loads, walked by the lanes in parallel once
// per GL steps and handed out by shuffles.  COL: 0 live, 1 full offsets.
struct StepBlock {
  int pk, ppo, mo, out, in0, in1, in2, f;
  float h;
};
template <int COL>
__device__ __forceinline__ StepBlock load_block(const GenDev& G, int g) {
  StepBlock b;
  b.f = G.fstep[g];
  const int* F = G.fprog + b.f;
  const int nin = F[3];
  b.pk = F[0] | (nin << 8) | (nin > 0 ? F[11] << 16 : 0) | (nin > 1 ? F[14] << 20 : 0) | (nin > 2 ? F[17] << 24 : 0);
  b.ppo = F[5];
  b.mo = F[6];
  b.out = F[7 + COL];
  b.in0 = nin > 0 ? F[9 + COL] : 0;
  b.in1 = nin > 1 ? F[12 + COL] : 0;
  b.in2 = nin > 2 ? F[15 + COL] : 0;
  b.h = 0.f;
  return b;
}
template <int COL>
__device__ __forceinline__ StepBlock load_block(const GenDev& G, int g, const int8_t* s) {
  StepBlock b = load_block<COL>(G, g);
  b.h = field_of(G, G.fprog[b.f + 1], G.fprog[b.f + 2], s);
  return b;
}
__device__ __forceinline__ Step block_step(const StepBlock& b, int j, int GL) {
  Step r;
  const int pk = __shfl_sync(0xffffffffu, b.pk, j, GL);
  r.m = pk & 255;
  r.nin = (pk >> 8) & 255;
  r.ppo = __shfl_sync(0xffffffffu, b.ppo, j, GL);
  r.mo = __shfl_sync(0xffffffffu, b.mo, j, GL);
  r.out = __shfl_sync(0xffffffffu, b.out, j, GL);
  r.in[0] = __shfl_sync(0xffffffffu, b.in0, j, GL);
  r.in[1] = __shfl_sync(0xffffffffu, b.in1, j, GL);
  r.in[2] = __shfl_sync(0xffffffffu, b.in2, j, GL);
  r.f = __shfl_sync(0xffffffffu, b.f, j, GL);
  r.h = __shfl_sync(0xffffffffu, b.h, j, GL);
  return r;
}

// Spins of the inputs of the group's step j.
__device__ __forceinline__ void next_widths(const StepBlock& b, int j, int (&kk)[3]) {
  const int pk = __shfl_sync(0xffffffffu, b.pk, j);
  kk[0] = (pk >> 16) & 15, kk[1] = (pk >> 20) & 15, kk[2] = (pk >> 24) & 15;
}

// Bond products of every step at this call's beta: one CTA per (step,
// instance), one thread per extended index.  A bond [[a,b],[b,a]] scaled by
// e^{-beta |J|} has entries 1 and e^{-2 beta |J|} (the latter where the two
// spins disagree for J >= 0, agree for J < 0).
__global__ void __launch_bounds__(256) general_pp_kernel(const InstDev* __restrict__ inst, const LaunchInfo li) {
  const int k = blockIdx.y;
  const InstDev& I = inst[k];
  if (I.kind != 2) return;
  const GenDev& G = I.gen;
  const int g = blockIdx.x;
  if (g >= G.n_steps) return;
  const StepRec r = step_at(G, g);
  const int E = 2 << r.m;
  const float beta = (float)li.beta[k];
  for (int ext = threadIdx.x; ext < E; ext += blockDim.x) {
    const int x = ext & ((1 << r.m) - 1), sg = ext >> r.m;
    float p = 1.f, d = 0.f;
    for (int j = 0; j < r.npair; ++j) {
      const float J = G.pairJ[r.pr[2 * j]], aj = fabsf(J);
      const bool same = ((x >> r.pr[2 * j + 1]) & 1) == sg;
      if (same != (J >= 0.f)) {
        p *= expf(-2.f * beta * aj);
        d -= 2.f * aj;
      }
    }
    G.pp[r.ppo + ext] = p;
    G.pp[G.n_pp + r.ppo + ext] = d;
  }
}

// Lanes per sample: a group of GL consecutive lanes (a power of two, at most
// 32, so that a group lies inside one warp) shares one sample; lane l of the
// group computes the table entries x = l, l + GL, ...  Every lane of a block
// runs the same program (invalid samples run on a dummy row), so the
// group-wide maximum and __syncwarp between steps see full warps.
// Row stride of the [entry][sample] tables: S samples plus 32 / GL floats,
// so that the GL consecutive entries written by a group and the 32 / GL
// samples of a warp fall in 32 different shared-memory banks.
__host__ __device__ __forceinline__ int gen_row_stride(int S, int GL) { return S + 32 / GL; }

__device__ __forceinline__ float group_max(float v, int GL) {
  for (int o = GL >> 1; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// The entries of one step's table for a sample (entry e of a table at A[e *
// RS]; with DB the beta-derivatives at dA[e * RS]): fv the eliminated spin's
// field factors, fr their beta-logarithmic derivatives, out the new table's
// offset, COL the input offsets' column (0 live, 1 full), NIN the number of
// input tables (-1: r.nin).  Returns the table's exponent; the table is
// written scaled by 2^-exponent, ZERO also clears Ab at its entries.
// A step is a chain of map, table and scale accesses whose latency sets the
// time, so a lane's entries are taken GEN_U at a time with every load of a
// batch independent, and tables of at most GEN_U entries a lane stay in
// registers until their scale is known (one table write instead of a write, a
// read and a write).
#define GEN_U 4
// Launches of more CTAs than this take one entry at a time in half of the
// registers instead: there the CTAs in flight hide the latency, and the batch's
// dropped entries are only instructions (n = 500 of degree 3, width 4, with
// d/dbeta: 32,768 samples in 1,024 CTAs 1,068 us four at a time, 653 one at a
// time; 4,096 samples in 256 CTAs 434 us four at a time, 526 one at a time).
#define GEN_FEW (2 * 152)
template <bool DB, int NIN, int COL, bool ZERO, int U0>
__device__ __forceinline__ int step_table(const Step& r, const GenDev& G, const float (&fv)[2], const float (&fr)[2],
                                          float* A, float* dA, float* Ab, int RS, int lane, int GL) {
  constexpr int U = DB && NIN >= 3 && U0 > 1 ? U0 / 2 : U0;  // within 128 registers
  const int out = r.out;
  const int M = 1 << r.m, E = 2 * M;
  const float* pp = G.pp + r.ppo;
  const float* pd = G.pp + G.n_pp + r.ppo;
  const unsigned short* mp = G.map + r.mo;
  const bool regs = M <= GL * U;
  float av[U], dv[U];
  float mx = 0.f;
  for (int x0 = lane; x0 < M; x0 += GL * U) {
    float p[U][2], rr[U][2];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = x0 + u * GL < M ? x0 + u * GL : x0;
#pragma unroll
      for (int sg = 0; sg < 2; ++sg) {
        p[u][sg] = pp[x | (sg << r.m)];
        rr[u][sg] = DB ? pd[x | (sg << r.m)] : 0.f;
      }
    }
    if constexpr (NIN >= 0) {
      float val[NIN > 0 ? NIN : 1][U][2], dval[NIN > 0 ? NIN : 1][U][2];
#pragma unroll
      for (int i = 0; i < NIN; ++i)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int x = x0 + u * GL < M ? x0 + u * GL : x0;
#pragma unroll
          for (int sg = 0; sg < 2; ++sg) {
            const int q = (r.in[i] + mp[i * E + (x | (sg << r.m))]) * RS;
            val[i][u][sg] = A[q];
            if (DB) dval[i][u][sg] = dA[q];
          }
        }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        // no divisions for what is dropped (M and GL are powers of two: the same for all lanes with an entry)
        if (DB && u * GL >= M) continue;
#pragma unroll
        for (int sg = 0; sg < 2; ++sg) {
          p[u][sg] = fv[sg] * p[u][sg];
          if (DB) rr[u][sg] = fr[sg] + rr[u][sg];
#pragma unroll
          for (int i = 0; i < NIN; ++i) {
            p[u][sg] *= val[i][u][sg];
            if (DB) rr[u][sg] += dval[i][u][sg] / val[i][u][sg];
          }
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int x = x0 + u * GL;
        if (u * GL >= M) continue;
#pragma unroll
        for (int sg = 0; sg < 2; ++sg) {
          p[u][sg] = fv[sg] * p[u][sg];
          if (DB) rr[u][sg] = fr[sg] + rr[u][sg];
          for (int i = 0; i < r.nin; ++i) {
            const int q = (G.fprog[r.f + 9 + 3 * i + COL] + mp[i * E + (x | (sg << r.m))]) * RS;
            const float v = A[q];
            p[u][sg] *= v;
            if (DB) rr[u][sg] += dA[q] / v;
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = x0 + u * GL;
      av[u] = dv[u] = 0.f;
      if (u * GL >= M) continue;
      av[u] = __fadd_rn(p[u][0], p[u][1]);  // the products' own rounding: not contracted into the last one
      if (DB) dv[u] = fmaf(p[u][1], rr[u][1], p[u][0] * rr[u][0]);
      mx = fmaxf(mx, av[u]);
      if (!regs) {
        A[(out + x) * RS] = av[u];
        if (DB) dA[(out + x) * RS] = dv[u];
      }
    }
  }
  mx = group_max(mx, GL);
  const int e = exponent_of(mx);
  const float sc = pow2i(-e);
  if (regs) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = lane + u * GL;
      if (x >= M) continue;
      A[(out + x) * RS] = av[u] * sc;
      if (DB) dA[(out + x) * RS] = dv[u] * sc;
      if (ZERO) Ab[(out + x) * RS] = 0.f;
    }
  } else {
#pragma unroll 4
    for (int x = lane; x < M; x += GL) {
      A[(out + x) * RS] *= sc;
      if (DB) dA[(out + x) * RS] *= sc;
      if (ZERO) Ab[(out + x) * RS] = 0.f;
    }
  }
  return e;
}

template <bool DB, int COL, bool ZERO, int U0>
__device__ __forceinline__ int step_table_any(const Step& r, const GenDev& G, const float (&fv)[2],
                                              const float (&fr)[2], float* A, float* dA, float* Ab, int RS, int lane,
                                              int GL) {
  switch (r.nin) {  // the same for every lane
    case 0: return step_table<DB, 0, COL, ZERO, U0>(r, G, fv, fr, A, dA, Ab, RS, lane, GL);
    case 1: return step_table<DB, 1, COL, ZERO, U0>(r, G, fv, fr, A, dA, Ab, RS, lane, GL);
    case 2: return step_table<DB, 2, COL, ZERO, U0>(r, G, fv, fr, A, dA, Ab, RS, lane, GL);
    case 3: return step_table<DB, 3, COL, ZERO, U0>(r, G, fv, fr, A, dA, Ab, RS, lane, GL);
    default: return step_table<DB, -1, COL, ZERO, U0>(r, G, fv, fr, A, dA, Ab, RS, lane, GL);
  }
}

// Component c for the sample whose tables start at A; forward, live offsets.
// Adds log Z_c (and with DB its beta-derivative) to lz / dl on lane 0 of the
// group.
template <bool DB, int U0>
__device__ __forceinline__ void run_component(const GenDev& G, int c, const int8_t* s, float* A, float* dA, int RS,
                                              int lane, int GL, float beta, double& lz, double& dl) {
  const int* H = G.fprog + G.fhdr[c];
  const int nsteps = H[0], fin = H[1];
  const int g0 = G.comp_step0[c];
  // log-scale terms of the component: the power-of-two scales add up exactly
  // as an integer, the field offsets |h_v| in a compensated FP32 sum (Kahan),
  // both added to the FP64 result once per component
  int esum = 0;
  float hs = 0.f, hc = 0.f;
  StepBlock blk;
  for (int st = 0; st < nsteps; ++st) {
    const int j = st & (GL - 1);
    if (j == 0) blk = load_block<0>(G, g0 + min(st + lane, nsteps - 1), s);
    const Step r = block_step(blk, j, GL);
    const float h = r.h, ah = fabsf(h);
    {
      const float y = ah - hc;
      const float t2 = hs + y;
      hc = (t2 - hs) - y;
      hs = t2;
    }
    const float fv[2] = {expf(beta * (h - ah)), expf(beta * (-h - ah))};
    const float fr[2] = {h - ah, -h - ah};
    esum += step_table_any<DB, 0, false, U0>(r, G, fv, fr, A, dA, nullptr, RS, lane, GL);
    __syncwarp();
  }
  if (lane == 0) {
    const double hsum = (double)hs - (double)hc;
    const float z = A[fin * RS];
    lz += (double)beta * hsum + (double)esum * 0.69314718055994530942 + (double)logf(z);
    if (DB) dl += hsum + (double)(dA[fin * RS] / z);
  }
}

// Boundary index of component c for spin row s: bit j set iff its j-th
// width-set neighbour (ctab boundary list) is -1.
__device__ __forceinline__ int boundary_index(const GenDev& G, const int* cr, const int8_t* s) {
  int idx = 0;
  for (int j = 0; j < cr[2]; ++j) idx |= (s[G.bpos[cr[3] + j]] < 0 ? 1 : 0) << j;
  return idx;
}

// Stage the spin rows of this CTA's samples in shared memory (rows of
// samples past the batch set to +1).
__device__ __forceinline__ void stage_spins(int8_t* ssp, const int8_t* gsp, int n_valid, int S, int D, int Dp) {
  for (int e = threadIdx.x; e < n_valid * D; e += blockDim.x) ssp[(e / D) * Dp + (e % D)] = gsp[e];
  for (int e = n_valid * Dp + threadIdx.x; e < S * Dp; e += blockDim.x) ssp[e] = 1;
}

// li.tile = samples per CTA (S); blockDim.x = S * GL.
template <bool DB, int U0>
__global__ void __launch_bounds__(128, U0 > 1 ? 4 : 8) general_kernel(const InstDev* __restrict__ inst,
                                                      const LaunchInfo li, int arena_floats, int GL,
                                                      const int8_t* __restrict__ spins,
                                                      double* __restrict__ logZR,
                                                      double* __restrict__ dbeta, float* __restrict__ garena) {
  extern __shared__ float sm[];
  const int k = find_inst(li, blockIdx.x);
  const InstDev& I = inst[k];
  if (I.kind != 2) return;
  const int S = li.tile, slot = threadIdx.x / GL, lane = threadIdx.x % GL;
  const int b0 = (blockIdx.x - li.tile_begin[k]) * S, b = b0 + slot;
  const float beta = (float)li.beta[k];
  const int D = I.D, Dp = padded_bytes(D);
  // tables [entry][sample] (rows of RS floats; then their beta-derivatives)
  // in shared memory, or for large arenas in this CTA's slice of a global
  // scratch buffer
  const int RS = gen_row_stride(S, GL);
  const size_t cta_floats = (size_t)arena_floats * RS * (DB ? 2 : 1);
  float* base = garena ? garena + (size_t)blockIdx.x * cta_floats : sm;
  float* A = base + slot;
  float* dA = A + (size_t)arena_floats * RS;
  int8_t* ssp = reinterpret_cast<int8_t*>(garena ? sm : sm + cta_floats);
  const GenDev& G = I.gen;
  const int n_valid = min(S, li.batch - b0);
  stage_spins(ssp, spins + I.spin_units * li.batch + (long long)b0 * D, n_valid, S, D, Dp);
  __syncthreads();
  const int8_t* s = ssp + slot * Dp;
  const bool tab = li.gen_tab && G.n_tab > 0 && G.n_tab <= li.batch;  // tables built for this call
  double lz = 0.0, dl = 0.0;
  for (int c = 0; c < G.n_comp; ++c) {
    const int* cr = G.ctab + 5 * c;
    if (tab && cr[4] >= 0) {  // a tabulated component: one lookup
      const int x = boundary_index(G, cr, s);
      lz += G.tab_lz[cr[4] + x];
      if (DB) dl += G.tab_db[cr[4] + x];
    } else {
      run_component<DB, U0>(G, c, s, A, dA, RS, lane, GL, beta, lz, dl);
    }
  }
  if (lane != 0 || b >= li.batch) return;
  float e1 = 0.f;
  for (int e = 0; e < I.n_ww; ++e) {
    const EdgeWW q = I.ww[e];
    e1 = fmaf(q.J, (float)(s[q.a] * s[q.b]), e1);
  }
  const double chf = G.c_hat;
  const long long o = (long long)k * li.batch + b;
  if (logZR) logZR[o] = lz + li.beta[k] * (chf + (double)e1);
  if (DB) dbeta[o] = dl + chf + (double)e1;
}

// ---------------------------------------------------------------------------
// The same contraction with lane = sample: a CTA takes 32 samples, its W warps
// share out each table's entries (warp w takes x = w, w + W, ...), tables are
// [entry][32 samples].  Every index (step record, map, bond product) is then
// the same for a warp's lanes and every table access one 128-byte row, where
// the lane-group form spends a warp's instructions on 32 / GL samples and, on
// the many small tables, leaves most lanes idle: 426 M warp instructions against
// 199 M for 4,096 samples of the n = 500 graph.  Costs two barriers a step.
// Bound by the steps' dependent chain: one CTA lasts ~400 steps whatever the
// batch.  Each entry's arithmetic, and so every result, is that of step_table.
// ---------------------------------------------------------------------------
#define G2_MAXW 8
// floats of a CTA: tables, fields of every step, and with d/dbeta the tables'
// derivatives
__host__ __device__ __forceinline__ size_t g2_main_floats(int arena, int steps) { return (size_t)(arena + steps) * 32; }

// The entries x = el, el + W, ... of a step's table, the table's maximum taken
// over the CTA's warps (red: two buffers of [warps][32], used in turn).
template <bool DB, int NIN, int COL, bool ZERO>
__device__ __forceinline__ int step_rows(const Step& r, const GenDev& G, const float (&fv)[2], const float (&fr)[2],
                                         float* A, float* dA, float* Ab, int el, int W, int lane, float* red) {
  constexpr int U = DB && NIN >= 3 ? GEN_U / 2 : GEN_U;
  const int M = 1 << r.m, E = 2 * M;
  const float* pp = G.pp + r.ppo;
  const float* pd = G.pp + G.n_pp + r.ppo;
  const unsigned short* mp = G.map + r.mo;
  const bool regs = M <= W * U;
  float* out = A + r.out * 32;
  float* dout = DB ? dA + r.out * 32 : nullptr;
  float av[U], dv[U];
  float mx = 0.f;
  for (int x0 = el; x0 < M; x0 += W * U) {
    float p[U][2], rr[U][2];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = x0 + u * W < M ? x0 + u * W : x0;
#pragma unroll
      for (int sg = 0; sg < 2; ++sg) {
        p[u][sg] = __ldg(pp + (x | (sg << r.m)));
        rr[u][sg] = DB ? __ldg(pd + (x | (sg << r.m))) : 0.f;
      }
    }
    if constexpr (NIN >= 0) {
      float val[NIN > 0 ? NIN : 1][U][2], dval[NIN > 0 ? NIN : 1][U][2];
#pragma unroll
      for (int i = 0; i < NIN; ++i)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int x = x0 + u * W < M ? x0 + u * W : x0;
#pragma unroll
          for (int sg = 0; sg < 2; ++sg) {
            const int q = (r.in[i] + __ldg(mp + i * E + (x | (sg << r.m)))) * 32;
            val[i][u][sg] = A[q];
            if (DB) dval[i][u][sg] = dA[q];
          }
        }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (DB && x0 + u * W >= M) continue;  // no divisions for what is dropped (the same for the whole warp)
#pragma unroll
        for (int sg = 0; sg < 2; ++sg) {
          p[u][sg] = fv[sg] * p[u][sg];
          if (DB) rr[u][sg] = fr[sg] + rr[u][sg];
#pragma unroll
          for (int i = 0; i < NIN; ++i) {
            p[u][sg] *= val[i][u][sg];
            if (DB) rr[u][sg] += dval[i][u][sg] / val[i][u][sg];
          }
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int x = x0 + u * W;
        if (x >= M) continue;
#pragma unroll
        for (int sg = 0; sg < 2; ++sg) {
          p[u][sg] = fv[sg] * p[u][sg];
          if (DB) rr[u][sg] = fr[sg] + rr[u][sg];
          for (int i = 0; i < r.nin; ++i) {
            const int q = (G.fprog[r.f + 9 + 3 * i + COL] + mp[i * E + (x | (sg << r.m))]) * 32;
            const float v = A[q];
            p[u][sg] *= v;
            if (DB) rr[u][sg] += dA[q] / v;
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = x0 + u * W;
      av[u] = dv[u] = 0.f;
      if (x >= M) continue;
      av[u] = __fadd_rn(p[u][0], p[u][1]);  // the products' own rounding: not contracted into the last one
      if (DB) dv[u] = fmaf(p[u][1], rr[u][1], p[u][0] * rr[u][0]);
      mx = fmaxf(mx, av[u]);
      if (!regs) {
        out[x * 32] = av[u];
        if (DB) dout[x * 32] = dv[u];
      }
    }
  }
  if (W > 1) {
    red[el * 32 + lane] = mx;
    __syncthreads();
    mx = red[lane];
    const int nw = min(W, M);  // warps that held entries
    for (int w = 1; w < nw; ++w) mx = fmaxf(mx, red[w * 32 + lane]);
  }
  const int e = exponent_of(mx);
  const float sc = pow2i(-e);
  if (regs) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = el + u * W;
      if (x >= M) continue;
      out[x * 32] = av[u] * sc;
      if (DB) dout[x * 32] = dv[u] * sc;
      if (ZERO) Ab[(r.out + x) * 32] = 0.f;
    }
  } else {
#pragma unroll 4
    for (int x = el; x < M; x += W) {
      out[x * 32] *= sc;
      if (DB) dout[x * 32] *= sc;
      if (ZERO) Ab[(r.out + x) * 32] = 0.f;
    }
  }
  return e;
}
template <bool DB, int COL, bool ZERO>
__device__ __forceinline__ int step_rows_any(const Step& r, const GenDev& G, const float (&fv)[2],
                                             const float (&fr)[2], float* A, float* dA, float* Ab, int el, int W,
                                             int lane, float* red) {
  switch (r.nin) {
    case 0: return step_rows<DB, 0, COL, ZERO>(r, G, fv, fr, A, dA, Ab, el, W, lane, red);
    case 1: return step_rows<DB, 1, COL, ZERO>(r, G, fv, fr, A, dA, Ab, el, W, lane, red);
    case 2: return step_rows<DB, 2, COL, ZERO>(r, G, fv, fr, A, dA, Ab, el, W, lane, red);
    case 3: return step_rows<DB, 3, COL, ZERO>(r, G, fv, fr, A, dA, Ab, el, W, lane, red);
    default: return step_rows<DB, -1, COL, ZERO>(r, G, fv, fr, A, dA, Ab, el, W, lane, red);
  }
}

// The fields of component steps [g0, g0 + nsteps) into h[step * 32] (this
// sample's column), the steps shared out over the warps.
__device__ __forceinline__ void step_fields(const GenDev& G, int g0, int nsteps, const int8_t* s, float* h, int el,
                                            int W) {
#pragma unroll 2
  for (int st = el; st < nsteps; st += W) {
    const int* F = G.fprog + G.fstep[g0 + st];
    h[st * 32] = field_of(G, F[1], F[2], s);
  }
}

// A read that only brings its line into L1; landed() ends its wait.
__device__ __forceinline__ int touch(const void* p) {
  int v;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)3));
  return v;
}
__device__ __forceinline__ void landed(int v) { asm volatile("" ::"r"(v)); }

// li.tile = 32; place: bit 0 tables and fields in shared memory, bit 1 the
// derivatives too, else in this CTA's slice of gscr.
template <bool DB>
__global__ void __launch_bounds__(32 * G2_MAXW, 2) general_rows_kernel(const InstDev* __restrict__ inst,
                                                                       const LaunchInfo li, int arena, int steps,
                                                                       int place, const int8_t* __restrict__ spins,
                                                                       double* __restrict__ logZR,
                                                                       double* __restrict__ dbeta,
                                                                       float* __restrict__ gscr) {
  extern __shared__ float sm[];
  __shared__ float red[2][G2_MAXW * 32];
  const int k = find_inst(li, blockIdx.x);
  const InstDev& I = inst[k];
  if (I.kind != 2) return;
  const int lane = threadIdx.x & 31, el = threadIdx.x >> 5, W = blockDim.x >> 5;
  const int b0 = (blockIdx.x - li.tile_begin[k]) * 32, b = b0 + lane;
  const float beta = (float)li.beta[k];
  const int D = I.D, Dp = padded_bytes(D);
  const size_t mf = g2_main_floats(arena, steps), df = (size_t)arena * 32;
  const size_t per = ((place & 1) ? 0 : mf) + (DB && !(place & 2) ? df : 0);
  float* sp = sm;
  float* gp = gscr + (size_t)blockIdx.x * per;
  float* A;
  if (place & 1) A = sp, sp += mf;
  else A = gp, gp += mf;
  float* dA = nullptr;
  if (DB) {
    if (place & 2) dA = sp, sp += df;
    else dA = gp;
  }
  float* h = A + (size_t)arena * 32 + lane;
  A += lane;
  if (DB) dA += lane;
  int8_t* ssp = reinterpret_cast<int8_t*>(sp);
  const GenDev& G = I.gen;
  stage_spins(ssp, spins + I.spin_units * li.batch + (long long)b0 * D, min(32, li.batch - b0), 32, D, Dp);
  __syncthreads();
  const int8_t* s = ssp + lane * Dp;
  const bool tab = li.gen_tab && G.n_tab > 0 && G.n_tab <= li.batch;  // tables built for this call
  double lz = 0.0, dl = 0.0;
  int par = 0;
  for (int c = 0; c < G.n_comp; ++c) {
    const int* cr = G.ctab + 5 * c;
    if (tab && cr[4] >= 0) {  // a tabulated component: one lookup
      const int x = boundary_index(G, cr, s);
      lz += G.tab_lz[cr[4] + x];
      if (DB) dl += G.tab_db[cr[4] + x];
      continue;
    }
    const int* H = G.fprog + G.fhdr[c];
    const int nsteps = H[0], fin = H[1], g0 = G.comp_step0[c];
    step_fields(G, g0, nsteps, s, h, el, W);
    __syncthreads();
    int esum = 0;
    float hs = 0.f, hc = 0.f;  // as run_component
    StepBlock blk, nxt = load_block<0>(G, g0 + min(lane, nsteps - 1));
    for (int st = 0; st < nsteps; ++st) {
      const int j = st & 31;
      if (j == 0) {
        blk = nxt;
        nxt = load_block<0>(G, g0 + min(st + 32 + lane, nsteps - 1));
      }
      const Step r = block_step(blk, j, 32);
      const float hv = h[st * 32], ah = fabsf(hv);
      {
        const float y = ah - hc;
        const float t2 = hs + y;
        hc = (t2 - hs) - y;
        hs = t2;
      }
      const float fv[2] = {expf(beta * (hv - ah)), expf(beta * (-hv - ah))};
      const float fr[2] = {hv - ah, -hv - ah};
      esum += step_rows_any<DB, 0, false>(r, G, fv, fr, A, dA, nullptr, el, W, lane, red[par]);
      par ^= 1;
      __syncthreads();
    }
    const double hsum = (double)hs - (double)hc;
    const float z = A[fin * 32];
    lz += (double)beta * hsum + (double)esum * 0.69314718055994530942 + (double)logf(z);
    if (DB) dl += hsum + (double)(dA[fin * 32] / z);
    __syncthreads();  // the tables and fields are free for the next component
  }
  if (el != 0 || b >= li.batch) return;
  float e1 = 0.f;
  for (int e = 0; e < I.n_ww; ++e) {
    const EdgeWW q = I.ww[e];
    e1 = fmaf(q.J, (float)(s[q.a] * s[q.b]), e1);
  }
  const double chf = G.c_hat;
  const long long o = (long long)k * li.batch + b;
  if (logZR) logZR[o] = lz + li.beta[k] * (chf + (double)e1);
  if (DB) dbeta[o] = dl + chf + (double)e1;
}

// The tables of the tabulated components (at most TNVAN_TAB_MAX_K width-set
// neighbours): group g of instance k takes entry g of the concatenated
// tables, i.e. one component c and one boundary configuration x, sets the
// boundary spins of a spin row from the bits of x (the other spins do not
// enter c) and runs c's program alone, so that tab_lz[toff_c + x] = log Z_c
// and tab_db[..] its beta-derivative.  Built per call (they depend on beta)
// when they are smaller than the batch.
template <bool DB>
__global__ void __launch_bounds__(128) general_tab_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
                                                          int arena_floats, int GL, float* __restrict__ garena) {
  extern __shared__ float sm[];
  const int k = blockIdx.y;
  const InstDev& I = inst[k];
  if (I.kind != 2) return;
  const GenDev& G = I.gen;
  if (G.n_tab == 0 || G.n_tab > li.batch) return;
  const int S = li.tile, slot = threadIdx.x / GL, lane = threadIdx.x % GL;
  const int g = blockIdx.x * S + slot;
  if (blockIdx.x * S >= G.n_tab) return;  // whole CTA idle (uniform)
  const float beta = (float)li.beta[k];
  const int D = I.D, Dp = padded_bytes(D);
  const int RS = gen_row_stride(S, GL);
  const size_t cta_floats = (size_t)arena_floats * RS * (DB ? 2 : 1);
  float* base = garena ? garena + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * cta_floats : sm;
  float* A = base + slot;
  float* dA = A + (size_t)arena_floats * RS;
  int8_t* ssp = reinterpret_cast<int8_t*>(garena ? sm : sm + cta_floats);
  int8_t* s = ssp + slot * Dp;
  for (int j = lane; j < D; j += GL) s[j] = 1;
  __syncwarp();
  // which tabulated component and configuration (entries past the tables
  // run the first tabulated component on the all-up row, unwritten)
  int c = -1, x = 0;
  for (int j = 0; j < G.n_tabc; ++j) {
    const int* cr = G.ctab + 5 * G.tabc[j];
    if (g >= cr[4] && g < cr[4] + (1 << cr[2])) {
      c = G.tabc[j];
      x = g - cr[4];
      break;
    }
  }
  const bool live = c >= 0;
  // every group of a warp must run the same component (shuffles, syncwarp):
  // the components of one warp's entries may differ, so a warp walks the
  // distinct components of its groups in turn
  const unsigned wmask = 0xffffffffu;
  int cc = live ? c : G.tabc[0];
  __syncwarp();
  for (;;) {
    // the smallest component index still to run in this warp
    int want = cc;
    for (int o = 16; o > 0; o >>= 1) want = min(want, __shfl_xor_sync(wmask, want, o));
    if (want == INT_MAX) break;
    const bool mine = cc == want;
    const int* cr = G.ctab + 5 * want;
    if (mine && live && lane == 0)
      for (int j = 0; j < cr[2]; ++j) s[G.bpos[cr[3] + j]] = ((x >> j) & 1) ? -1 : 1;
    __syncwarp();
    double lz = 0.0, dl = 0.0;
    run_component<DB, GEN_U>(G, want, s, A, dA, RS, lane, GL, beta, lz, dl);
    if (mine && live && lane == 0) {
      G.tab_lz[g] = lz;
      if (DB) G.tab_db[g] = dl;
    }
    if (mine) cc = INT_MAX;
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// Reverse mode: d ln Z_c / d J_e for the bonds inside a component (beta <r r'>)
// and its bonds to the width set (beta s_w <r>).  Per component the steps run
// forward storing every (renormalised) table A_t and its scale 2^-e_t (full
// offsets); then backwards carrying adjoints Abar = d ln Z / d A of each table
// entry, starting from 1 / A_final.  For step t with product terms
// term(x, sigma) (field factor, bond factors, input tables):
//   g(x, sigma)       = Abar_t[x] 2^-e_t term(x, sigma)
//   Abar_in[idx]     += g / A_in[idx]
//   d lnZ / d J_bond += beta sum g sigma sigma_u,  d lnZ / d J_field += beta s_w sum g sigma.
// The input adjoints are gathered per input entry (inverse maps) from the
// step's stored g values, in a fixed order.  Bond sums are warp-reduced (over
// samples and lanes) into per-warp shared rows, added in warp order into one
// row per CTA, and the rows added per instance in a fixed order: the result
// does not depend on scheduling.
// ---------------------------------------------------------------------------
// Four bond sums at once (their shuffles overlap).
__device__ __forceinline__ void acc_edges(float* acc_w, const int (&e)[4], float (&v)[4], bool lane0) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (lane0 && e[j] >= 0) acc_w[e[j]] += v[j];
}

// The product terms of one step in the reverse sweep: g(x, sigma) into gb, its
// sums with sigma (gs) and with sigma sigma_u of the first NPU bonds (gp), in
// the order of x; loads GEN_U entries at a time.
template <int NIN, int NPU, int U0>
__device__ __forceinline__ void step_g(const Step& r, const GenDev& G, const float (&fv)[2], const float* A,
                                       const float* Ab, float* gb, int RS, float scl, const int* pos, int np,
                                       int lane, int GL, float& gs, float (&gp)[TNVAN_MAX_ELIM_W]) {
  const int out = r.out;
  const int M = 1 << r.m, E = 2 * M;
  const float* pp = G.pp + r.ppo;
  const unsigned short* mp = G.map + r.mo;
  for (int x0 = lane; x0 < M; x0 += GL * U0) {
    float p[U0][2], abx[U0];
#pragma unroll
    for (int u = 0; u < U0; ++u) {
      const int x = x0 + u * GL < M ? x0 + u * GL : x0;
      abx[u] = Ab[(out + x) * RS];
#pragma unroll
      for (int sg = 0; sg < 2; ++sg) p[u][sg] = pp[x | (sg << r.m)];
    }
    if constexpr (NIN >= 0) {
      float val[NIN > 0 ? NIN : 1][U0][2];
#pragma unroll
      for (int i = 0; i < NIN; ++i)
#pragma unroll
        for (int u = 0; u < U0; ++u) {
          const int x = x0 + u * GL < M ? x0 + u * GL : x0;
#pragma unroll
          for (int sg = 0; sg < 2; ++sg) val[i][u][sg] = A[(r.in[i] + mp[i * E + (x | (sg << r.m))]) * RS];
        }
#pragma unroll
      for (int u = 0; u < U0; ++u) {
#pragma unroll
        for (int sg = 0; sg < 2; ++sg) {
          p[u][sg] = fv[sg] * p[u][sg];
#pragma unroll
          for (int i = 0; i < NIN; ++i) p[u][sg] *= val[i][u][sg];
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < U0; ++u) {
        const int x = x0 + u * GL;
        if (u * GL >= M) continue;
#pragma unroll
        for (int sg = 0; sg < 2; ++sg) {
          p[u][sg] = fv[sg] * p[u][sg];
          for (int i = 0; i < r.nin; ++i) p[u][sg] *= A[(G.fprog[r.f + 9 + 3 * i + 1] + mp[i * E + (x | (sg << r.m))]) * RS];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U0; ++u) {
      const int x = x0 + u * GL;
      if (u * GL >= M) continue;
      const float ab = abx[u] * scl;
#pragma unroll
      for (int sg = 0; sg < 2; ++sg) {
        const float g = ab * p[u][sg];
        gb[(x | (sg << r.m)) * RS] = g;
        gs = fmaf(g, sg ? -1.f : 1.f, gs);
#pragma unroll
        for (int j = 0; j < NPU; ++j)
          if (j < np) gp[j] = fmaf(g, (((x >> pos[j]) & 1) == sg) ? 1.f : -1.f, gp[j]);
      }
    }
  }
}
template <int NPU, int U0>
__device__ __forceinline__ void step_g_any(const Step& r, const GenDev& G, const float (&fv)[2], const float* A,
                                           const float* Ab, float* gb, int RS, float scl, const int* pos, int np,
                                           int lane, int GL, float& gs, float (&gp)[TNVAN_MAX_ELIM_W]) {
  switch (r.nin) {  // the same for every lane
    case 0: step_g<0, NPU, U0>(r, G, fv, A, Ab, gb, RS, scl, pos, np, lane, GL, gs, gp); break;
    case 1: step_g<1, NPU, U0>(r, G, fv, A, Ab, gb, RS, scl, pos, np, lane, GL, gs, gp); break;
    case 2: step_g<2, NPU, U0>(r, G, fv, A, Ab, gb, RS, scl, pos, np, lane, GL, gs, gp); break;
    default: step_g<-1, NPU, U0>(r, G, fv, A, Ab, gb, RS, scl, pos, np, lane, GL, gs, gp); break;
  }
}

template <int U0>
__global__ void __launch_bounds__(128, U0 > 1 ? 4 : 8) general_dJ_kernel(const InstDev* __restrict__ inst,
                                                         const LaunchInfo li, int arena_floats, int max_steps,
                                                         int gmax, int GL, const int8_t* __restrict__ spins,
                                                         float* __restrict__ part, int part_stride,
                                                         float* __restrict__ garena) {
  extern __shared__ float sm[];
  const int k = find_inst(li, blockIdx.x);
  const InstDev& I = inst[k];
  if (I.kind != 2) return;
  const int S = li.tile, slot = threadIdx.x / GL, lane = threadIdx.x % GL;
  const int b0 = (blockIdx.x - li.tile_begin[k]) * S, b = b0 + slot;
  const float beta = (float)li.beta[k];
  const int D = I.D, Dp = padded_bytes(D);
  // tables, adjoints, scales and the step's g values, each [entry][sample]
  // (rows of RS floats), in shared memory or for large arenas in this CTA's
  // slice of a global scratch buffer
  const int RS = gen_row_stride(S, GL);
  const size_t cta_floats = (size_t)(2 * arena_floats + max_steps + gmax) * RS;
  float* base = garena ? garena + (size_t)blockIdx.x * cta_floats : sm;
  float* A = base + slot;                          // [arena]
  float* Ab = A + (size_t)arena_floats * RS;       // [arena] adjoints
  float* sc = Ab + (size_t)arena_floats * RS;      // [max_steps] scales 2^-e
  float* gb = sc + (size_t)max_steps * RS;         // [gmax] g of the current step
  const int ne4 = (I.n_edges + 3) & ~3, nw = blockDim.x >> 5;
  float* acc = garena ? sm : sm + cta_floats;  // [warps][n_edges]
  float* acc_w = acc + (threadIdx.x >> 5) * ne4;
  int8_t* ssp = reinterpret_cast<int8_t*>(acc + nw * ne4);
  const GenDev& G = I.gen;
  for (int e = threadIdx.x; e < nw * ne4; e += blockDim.x) acc[e] = 0.f;
  const int n_valid = min(S, li.batch - b0);
  stage_spins(ssp, spins + I.spin_units * li.batch + (long long)b0 * D, n_valid, S, D, Dp);
  __syncthreads();
  const bool valid = b < li.batch;
  const bool lane0 = (threadIdx.x & 31) == 0;
  const int8_t* s = ssp + slot * Dp;
  // per-sample weight of the bond sums (importance multipliers when given)
  const float wscale =
      valid ? beta / (float)li.batch * (li.wmul ? li.wmul[(long long)k * li.batch + b] : 1.f) : 0.f;
  for (int c = 0; c < G.n_comp; ++c) {
    const int* H = G.fprog + G.fhdr[c];
    const int nsteps = H[0], fin = H[2];
    const int g0 = G.comp_step0[c];
    // forward: tables and their scales
    const float fr[2] = {0.f, 0.f};
    StepBlock blk;
    for (int st = 0; st < nsteps; ++st) {
      const int j = st & (GL - 1);
      if (j == 0) blk = load_block<1>(G, g0 + min(st + lane, nsteps - 1), s);
      const Step r = block_step(blk, j, GL);
      const float h = r.h, ah = fabsf(h);
      const float fv[2] = {expf(beta * (h - ah)), expf(beta * (-h - ah))};
      const int e = step_table_any<false, 1, true, U0>(r, G, fv, fr, A, nullptr, Ab, RS, lane, GL);
      if (lane == 0) sc[st * RS] = pow2i(-e);
      __syncwarp();
    }
    if (lane == 0) Ab[fin * RS] = 1.f / A[fin * RS];
    __syncwarp();
    // backward
    for (int st = nsteps - 1, j0 = 0; st >= 0; --st, ++j0) {
      const int jb = j0 & (GL - 1);
      if (jb == 0) blk = load_block<1>(G, g0 + max(st - lane, 0), s);
      const Step r = block_step(blk, jb, GL);
      const int* F = G.fprog + r.f;
      const int fb = F[1], fc = F[2], npair = F[4];
      const int* pr = F + 9 + 3 * r.nin;
      const float h = r.h, ah = fabsf(h);
      const float fv[2] = {expf(beta * (h - ah)), expf(beta * (-h - ah))};
      const int E = 2 << r.m;
      const unsigned short* mp = G.map + r.mo;
      const float scl = sc[st * RS];
      constexpr int MW = TNVAN_MAX_ELIM_W;
      const int np = min(npair, MW);  // at most MW neighbours remain
      int pos[MW];
#pragma unroll
      for (int j = 0; j < MW; ++j) pos[j] = j < np ? pr[2 * j + 1] : 0;
      float gs = 0.f;       // sum g sigma_v
      float gp[MW];         // sum g sigma_v sigma_u per pair
#pragma unroll
      for (int j = 0; j < MW; ++j) gp[j] = 0.f;
      if (np <= 4) step_g_any<4, U0>(r, G, fv, A, Ab, gb, RS, scl, pos, np, lane, GL, gs, gp);
      else step_g_any<MW, U0>(r, G, fv, A, Ab, gb, RS, scl, pos, np, lane, GL, gs, gp);
      __syncwarp();
      // input adjoints: each entry gathers the g of the extended indices that
      // read it (inverse map), lanes split the entries
      for (int i = 0; i < r.nin; ++i) {
        const int in = F[9 + 3 * i + 1], kk = F[9 + 3 * i + 2];
        const int R = E >> kk;
        const unsigned short* inv = mp + (r.nin + i) * E;
#pragma unroll 2
        for (int e = lane; e < (1 << kk); e += GL) {
          const float av = A[(in + e) * RS];
          float sum = 0.f;
          for (int f = 0; f + 4 <= R; f += 4) {  // in index order, four loads in flight
            float q[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) q[j] = gb[inv[e * R + f + j] * RS];
#pragma unroll
            for (int j = 0; j < 4; ++j) sum += q[j];
          }
          if (R < 4)
            for (int f = 0; f < R; ++f) sum += gb[inv[e * R + f] * RS];
          if (av > 0.f) Ab[(in + e) * RS] += sum / av;
        }
      }
      for (int f0 = 0; f0 < fc; f0 += 4) {
        int ee[4];
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int f = fb + f0 + j;
          ee[j] = f0 + j < fc ? G.fld[2 * f + 1] : -1;
          v[j] = f0 + j < fc ? wscale * gs * (float)s[G.fld[2 * f]] : 0.f;
        }
        acc_edges(acc_w, ee, v, lane0);
      }
#pragma unroll
      for (int p0 = 0; p0 < MW; p0 += 4) {
        if (p0 >= np) break;
        int ee[4];
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          ee[j] = p0 + j < np ? G.pairE[pr[2 * (p0 + j)]] : -1;
          v[j] = wscale * gp[p0 + j];
        }
        acc_edges(acc_w, ee, v, lane0);
      }
      __syncwarp();
    }
  }
  __syncthreads();
  float* row = part + (long long)blockIdx.x * part_stride;
  for (int e = threadIdx.x; e < I.n_edges; e += blockDim.x) {
    float v = 0.f;
    for (int w = 0; w < nw; ++w) v += acc[w * ne4 + e];
    row[e] = v;
  }
}

// ---------------------------------------------------------------------------
// The reverse sweep with lane = sample (see general_rows_kernel), 32 samples
// and 16 warps per CTA.  general_dJ_kernel's order of every sum is kept, so
// d/dJ has the same bits in both forms: a bond's sum over a step's entries is
// made of W (4 or 8, that kernel's lanes per sample) chains x = w, w + W, ...,
// each added over the 32 / W samples of a group, then over the chains by the
// same tree, the groups' rows in turn into one row per 128 / W samples.
//
// Tables and adjoints (1.3 MB for 32 samples of the n = 500 graph) stay in
// global memory, i.e. L2, so a step is a chain of dependent L2 reads: record ->
// maps -> tables -> g -> adjoints.  The next step's record, bond products, maps
// and table rows are therefore read into L1 a step ahead (touch), and all 16
// warps share out the extended indices, the bonds and the gathered entries.
// 4,096 samples of the n = 500 graph, width 8: 1,769 us against 2,380 in the
// lane-group form; without the reads ahead and with W warps only, 2,287.
// ---------------------------------------------------------------------------
#define G2_DJ_WARPS 16

// Touch what step r will read: threads 0-31 bond products, 32-127 n_maps maps
// of its extended indices, 128 and 129 its record, and each thread a row of its
// inputs' tables (T) and, with ADJ, of their adjoints.
struct Touched {
  int a, b, c;
};
template <bool ADJ>
__device__ __forceinline__ Touched touch_step(const GenDev& G, const Step& r, const int (&kk)[3], int n_maps,
                                              const float* A, const float* Ab, int t) {
  const int E = 2 << r.m;
  Touched v = {0, 0, 0};
  if (t < 32) {
    if (t * 32 < E + 32) v.a = touch(G.pp + r.ppo + min(t * 32, E - 1));
  } else if (t < 128) {
    const int nm = n_maps * E, o = (t - 32) * 64;
    if (nm > 0 && o < nm + 64) v.a = touch(G.map + r.mo + min(o, nm - 1));
  } else if (ADJ && t < 130) {
    v.a = touch(G.fprog + r.f + (t == 128 ? 0 : 8));
  }
  int q = t;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (i >= r.nin) break;
    const int n = 1 << kk[i];
    if (q >= 0 && q < n) {
      v.b = touch(A + (r.in[i] + q) * 32);
      if (ADJ) v.c = touch(Ab + (r.in[i] + q) * 32);
    }
    q -= n;
  }
  return v;
}

// g of the extended indices ext = w0, w0 + NW, ... of a step, into gb.
template <int NIN>
__device__ __forceinline__ void rows_g(const Step& r, const GenDev& G, const float (&fv)[2], const float* A,
                                       const float* Ab, float* gb, float scl, int w0, int NW) {
  const int M = 1 << r.m, E = 2 * M;
  const float* pp = G.pp + r.ppo;
  const unsigned short* mp = G.map + r.mo;
  for (int e0 = w0; e0 < E; e0 += NW * GEN_U) {
    float p[GEN_U], ab[GEN_U], val[NIN > 0 ? NIN : 1][GEN_U];
#pragma unroll
    for (int u = 0; u < GEN_U; ++u) {
      const int ext = e0 + u * NW;
      p[u] = ab[u] = 0.f;
#pragma unroll
      for (int i = 0; i < NIN; ++i) val[i][u] = 0.f;
      if (ext >= E) continue;
      p[u] = __ldg(pp + ext);
      ab[u] = Ab[(r.out + (ext & (M - 1))) * 32];
#pragma unroll
      for (int i = 0; i < NIN; ++i) val[i][u] = A[(r.in[i] + __ldg(mp + i * E + ext)) * 32];
    }
#pragma unroll
    for (int u = 0; u < GEN_U; ++u) {
      const int ext = e0 + u * NW;
      if (ext >= E) continue;
      float v = ((ext >> r.m) & 1 ? fv[1] : fv[0]) * p[u];
      if constexpr (NIN >= 0) {
#pragma unroll
        for (int i = 0; i < NIN; ++i) v *= val[i][u];
      } else {
        for (int i = 0; i < r.nin; ++i) v *= A[(G.fprog[r.f + 9 + 3 * i + 1] + mp[i * E + ext]) * 32];
      }
      gb[ext * 32] = (ab[u] * scl) * v;
    }
  }
}

// A bond value's sum over the samples of each group of 32 / W: at the groups'
// first lanes.
template <int W>
__device__ __forceinline__ float group_samples(float v) {
#pragma unroll
  for (int o = 16; o >= W; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o / W);
  return v;
}

// The W chains of a step's sum of g times a sign: that of the eliminated spin
// (pos < 0), or of its product with out-scope spin pos.
template <int W>
__device__ __forceinline__ void bond_chains(const float* gb, int m, int pos, float (&v)[W]) {
  const int M = 1 << m;
#pragma unroll
  for (int w = 0; w < W; ++w) v[w] = 0.f;
  for (int x0 = 0; x0 < M; x0 += W) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const int x = x0 + w;
      if (x >= M) break;
      const int bit = pos < 0 ? 0 : (x >> pos) & 1;
      v[w] = fmaf(gb[x * 32], bit == 0 ? 1.f : -1.f, v[w]);
      v[w] = fmaf(gb[(x + M) * 32], bit == 1 ? 1.f : -1.f, v[w]);
    }
  }
}
// The chains, each times mul and added over the groups' samples, added up; into
// edge e of each group's row (ne4 floats).
template <int W>
__device__ __forceinline__ void bond_add(const float (&v)[W], float wscale, float sgn, bool signed_, float* acc,
                                         int ne4, int e, int lane) {
  float u[W];
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const float q = wscale * v[w];
    u[w] = group_samples<W>(signed_ ? q * sgn : q);
  }
  if (W == 8) {
#pragma unroll
    for (int w = 0; w < 4; ++w) u[w] += u[w + W / 2];
  }
  u[0] += u[2];
  u[1] += u[3];
  const float sum = u[0] + u[1];
  if (e >= 0 && (lane & (32 / W - 1)) == 0) acc[lane / (32 / W) * ne4 + e] += sum;
}

// Dynamic shared memory: g values [gmax][32], bond sums [W][n_edges], spins.
// Tables, adjoints, scales and fields ((2 arena + 2 steps) x 32 floats) in this
// CTA's slice of gscr.
template <int W>
__global__ void __launch_bounds__(32 * G2_DJ_WARPS, 1) general_rows_dJ_kernel(
    const InstDev* __restrict__ inst, const LaunchInfo li, int arena, int steps, int gmax,
    const int8_t* __restrict__ spins, float* __restrict__ part, int part_stride, float* __restrict__ gscr) {
  extern __shared__ float sm[];
  __shared__ float red[2][G2_DJ_WARPS * 32];
  const int k = find_inst(li, blockIdx.x);
  const InstDev& I = inst[k];
  if (I.kind != 2) return;
  constexpr int NW = G2_DJ_WARPS;
  const int t = threadIdx.x, lane = t & 31, wi = t >> 5;
  const int c_idx = blockIdx.x - li.tile_begin[k];
  const int b0 = c_idx * 32, b = b0 + lane;
  const float beta = (float)li.beta[k];
  const int D = I.D, Dp = padded_bytes(D), ne = I.n_edges, ne4 = (ne + 3) & ~3;
  float* A0 = gscr + (size_t)blockIdx.x * (size_t)(2 * arena + 2 * steps) * 32;
  float* A = A0 + lane;
  float* Ab0 = A0 + (size_t)arena * 32;
  float* Ab = Ab0 + lane;
  float* sc = Ab + (size_t)arena * 32;
  float* h = sc + (size_t)steps * 32;
  float* gb = sm + lane;
  float* acc = sm + gmax * 32;  // [W groups][ne4]
  int8_t* ssp = reinterpret_cast<int8_t*>(acc + W * ne4);
  const GenDev& G = I.gen;
  for (int e = t; e < W * ne4; e += 32 * NW) acc[e] = 0.f;
  stage_spins(ssp, spins + I.spin_units * li.batch + (long long)b0 * D, min(32, li.batch - b0), 32, D, Dp);
  __syncthreads();
  const int8_t* s = ssp + lane * Dp;
  // per-sample weight of the bond sums (importance multipliers when given)
  const float wscale =
      b < li.batch ? beta / (float)li.batch * (li.wmul ? li.wmul[(long long)k * li.batch + b] : 1.f) : 0.f;
  int par = 0;
  for (int c = 0; c < G.n_comp; ++c) {
    const int* H = G.fprog + G.fhdr[c];
    const int nsteps = H[0], fin = H[2], g0 = G.comp_step0[c];
    step_fields(G, g0, nsteps, s, h, wi, NW);
    __syncthreads();
    const float fr[2] = {0.f, 0.f};
    int kk[3];
    {
      StepBlock blk = load_block<1>(G, g0 + min(lane, nsteps - 1)), nxt = blk;
      float hv = h[0];
      for (int st = 0; st < nsteps; ++st) {
        const int j = st & 31;
        if (j == 0) {
          blk = nxt;
          nxt = load_block<1>(G, g0 + min(st + 32 + lane, nsteps - 1));
        }
        const Step r = block_step(blk, j, 32);
        const Step rn = block_step(j == 31 ? nxt : blk, (j + 1) & 31, 32);
        next_widths(j == 31 ? nxt : blk, (j + 1) & 31, kk);
        const float hn = h[min(st + 1, nsteps - 1) * 32], ah = fabsf(hv);
        const Touched tc = touch_step<false>(G, rn, kk, rn.nin, A0, Ab0, t);
        const float fv[2] = {expf(beta * (hv - ah)), expf(beta * (-hv - ah))};
        const int e = step_rows_any<false, 1, true>(r, G, fv, fr, A, nullptr, Ab, wi, NW, lane, red[par]);
        par ^= 1;
        if (wi == 0) sc[st * 32] = pow2i(-e);
        hv = hn;
        landed(tc.a), landed(tc.b);
        __syncthreads();
      }
    }
    if (wi == 0) Ab[fin * 32] = 1.f / A[fin * 32];
    __syncthreads();
    StepBlock blk, nxt = load_block<1>(G, g0 + max(nsteps - 1 - lane, 0));
    float hv = h[(nsteps - 1) * 32], scl = sc[(nsteps - 1) * 32];
    for (int st = nsteps - 1, j0 = 0; st >= 0; --st, ++j0) {
      const int jb = j0 & 31;
      if (jb == 0) {
        blk = nxt;
        nxt = load_block<1>(G, g0 + max(st - 32 - lane, 0));
      }
      const Step r = block_step(blk, jb, 32);
      const Step rn = block_step(jb == 31 ? nxt : blk, (jb + 1) & 31, 32);
      next_widths(jb == 31 ? nxt : blk, (jb + 1) & 31, kk);
      const float hn = h[max(st - 1, 0) * 32], scn = sc[max(st - 1, 0) * 32], ah = fabsf(hv);
      const Touched tc = touch_step<true>(G, rn, kk, 2 * rn.nin, A0, Ab0, t);
      const int* F = G.fprog + r.f;
      const int fb = F[1], fc = F[2], np = min(F[4], TNVAN_MAX_ELIM_W);
      const int* pr = F + 9 + 3 * r.nin;
      const float fv[2] = {expf(beta * (hv - ah)), expf(beta * (-hv - ah))};
      switch (r.nin) {
        case 0: rows_g<0>(r, G, fv, A, Ab, gb, scl, wi, NW); break;
        case 1: rows_g<1>(r, G, fv, A, Ab, gb, scl, wi, NW); break;
        case 2: rows_g<2>(r, G, fv, A, Ab, gb, scl, wi, NW); break;
        default: rows_g<-1>(r, G, fv, A, Ab, gb, scl, wi, NW); break;
      }
      __syncthreads();
      // bonds, a warp each from the last warp on: one for the fields (if any),
      // one for each pair
      const int nq = np + (fc > 0);
      for (int q = NW - 1 - wi; q < nq; q += NW) {
        float v[W];
        const int j = q - (fc > 0);
        if (j < 0) {
          bond_chains<W>(gb, r.m, -1, v);
          for (int f = 0; f < fc; ++f)
            bond_add<W>(v, wscale, (float)s[G.fld[2 * (fb + f)]], true, acc, ne4, G.fld[2 * (fb + f) + 1], lane);
        } else {
          bond_chains<W>(gb, r.m, pr[2 * j + 1], v);
          bond_add<W>(v, wscale, 1.f, false, acc, ne4, G.pairE[pr[2 * j]], lane);
        }
      }
      // input adjoints: each entry gathers the g of the extended indices that read it
      const int E = 2 << r.m;
      const unsigned short* mp = G.map + r.mo;
      for (int i = 0; i < r.nin; ++i) {
        const int in = F[9 + 3 * i + 1], ki = F[9 + 3 * i + 2];
        const int R = E >> ki;
        const unsigned short* inv = mp + (r.nin + i) * E;
#pragma unroll 2
        for (int e = wi; e < (1 << ki); e += NW) {
          const float av = A[(in + e) * 32];
          float sum = 0.f;
          for (int f = 0; f + 4 <= R; f += 4) {  // in index order, four loads in flight
            float q[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) q[j] = gb[__ldg(inv + e * R + f + j) * 32];
#pragma unroll
            for (int j = 0; j < 4; ++j) sum += q[j];
          }
          if (R < 4)
            for (int f = 0; f < R; ++f) sum += gb[inv[e * R + f] * 32];
          if (av > 0.f) Ab[(in + e) * 32] += sum / av;
        }
      }
      hv = hn, scl = scn;
      landed(tc.a), landed(tc.b), landed(tc.c);
      __syncthreads();
    }
  }
  // one row per 128 / W samples: its four groups in turn
  const int rows = W / 4, n_rows = (li.batch + 128 / W - 1) / (128 / W);
  const long long row0 = (long long)k * n_rows + (long long)c_idx * rows;
  for (int q = 0; q < rows && c_idx * rows + q < n_rows; ++q) {
    float* row = part + (row0 + q) * part_stride;
    for (int e = t; e < ne; e += 32 * NW) {
      float v = 0.f;
      for (int w = 0; w < 4; ++w) v += acc[(4 * q + w) * ne4 + e];
      row[e] = v;
    }
  }
}

__global__ void general_dJ_reduce_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
                                         const float* __restrict__ part, int part_stride,
                                         double* __restrict__ dJ) {
  const int k = blockIdx.y;
  const InstDev& I = inst[k];
  if (I.kind != 2) return;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < I.n_edges; e += gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int c = li.tile_begin[k]; c < li.tile_begin[k + 1]; ++c) s += (double)part[(long long)c * part_stride + e];
    dJ[I.edge_off + e] += s;
  }
}

cudaError_t launch_general_pp(const InstDev* d_inst, const LaunchInfo& li, int max_steps, cudaStream_t s) {
  if (max_steps <= 0) return cudaSuccess;
  general_pp_kernel<<<dim3(max_steps, li.n_inst), 256, 0, s>>>(d_inst, li);
  return cudaGetLastError();
}

// per-sample floats: 2 * arena + steps + gmax (tables, adjoints, scales, g)
int general_dJ_smem_bytes(int per_sample, int D, int n_edges, int T, int GL, bool glob) {
  int w4 = (D + 3) / 4;
  if ((w4 & 1) == 0) ++w4;
  return (glob ? 0 : per_sample * gen_row_stride(T, GL) * 4) + (T * GL / 32) * ((n_edges + 3) & ~3) * 4 +
         T * 4 * w4;
}

size_t general_dJ_scratch_floats(int per_sample, int T, int GL, int nblk) {
  return (size_t)per_sample * gen_row_stride(T, GL) * nblk;
}

cudaError_t launch_general_dJ(const InstDev* d_inst, const LaunchInfo& li, int smem_bytes, int arena, int steps,
                              int gmax, int GL, const int8_t* spins, float* part, int part_stride, double* dJ,
                              float* garena, cudaStream_t s) {
  const int nblk = li.tile_begin[li.n_inst];
  if (nblk == 0) return cudaSuccess;
  auto kern = nblk <= GEN_FEW ? general_dJ_kernel<GEN_U> : general_dJ_kernel<1>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  kern<<<nblk, li.tile * GL, smem_bytes, s>>>(d_inst, li, arena, steps, gmax, GL, spins, part, part_stride, garena);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  general_dJ_reduce_kernel<<<dim3(4, li.n_inst), 256, 0, s>>>(d_inst, li, part, part_stride, dJ);
  return cudaGetLastError();
}

int general_rows_smem_bytes(int arena, int steps, int D, bool db, int place) {
  int w4 = (D + 3) / 4;
  if ((w4 & 1) == 0) ++w4;
  return (int)(4 * (((place & 1) ? g2_main_floats(arena, steps) : 0) + (db && (place & 2) ? (size_t)arena * 32 : 0))) +
         32 * 4 * w4;
}
size_t general_rows_scratch_floats(int arena, int steps, bool db, int place, int nblk) {
  return (((place & 1) ? 0 : g2_main_floats(arena, steps)) + (db && !(place & 2) ? (size_t)arena * 32 : 0)) * nblk;
}
cudaError_t launch_general_rows(const InstDev* d_inst, const LaunchInfo& li, int smem_bytes, int W, int arena,
                                int steps, int place, const int8_t* spins, double* logZR, double* dbeta, float* gscr,
                                cudaStream_t s) {
  const int nblk = li.tile_begin[li.n_inst];
  if (nblk == 0) return cudaSuccess;
  auto kern = dbeta ? general_rows_kernel<true> : general_rows_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  kern<<<nblk, 32 * W, smem_bytes, s>>>(d_inst, li, arena, steps, place, spins, logZR, dbeta, gscr);
  return cudaGetLastError();
}

int general_rows_dJ_smem_bytes(int D, int n_edges, int gmax, int W) {
  int w4 = (D + 3) / 4;
  if ((w4 & 1) == 0) ++w4;
  return 4 * (gmax * 32 + W * ((n_edges + 3) & ~3)) + 32 * 4 * w4;
}
size_t general_rows_dJ_scratch_floats(int arena, int steps, int nblk) {
  return (size_t)(2 * arena + 2 * steps) * 32 * nblk;
}
cudaError_t launch_general_rows_dJ(const InstDev* d_inst, const LaunchInfo& li, const LaunchInfo& lr, int smem_bytes,
                                   int W, int arena, int steps, int gmax, const int8_t* spins, float* part,
                                   int part_stride, double* dJ, float* gscr, cudaStream_t s) {
  const int nblk = li.tile_begin[li.n_inst];
  if (nblk == 0) return cudaSuccess;
  auto kern = W == 8 ? general_rows_dJ_kernel<8> : general_rows_dJ_kernel<4>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  kern<<<nblk, 32 * G2_DJ_WARPS, smem_bytes, s>>>(d_inst, li, arena, steps, gmax, spins, part, part_stride, gscr);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  general_dJ_reduce_kernel<<<dim3(4, lr.n_inst), 256, 0, s>>>(d_inst, lr, part, part_stride, dJ);
  return cudaGetLastError();
}

// The components' tables at this call's betas (li.gen_tab: the largest
// table; the contraction kernels then look them up).
cudaError_t launch_general_tables(const InstDev* d_inst, const LaunchInfo& li, int smem_bytes, bool db, int GL,
                                  float* garena, cudaStream_t s) {
  if (li.gen_tab <= 0) return cudaSuccess;
  const int arena = (int)(li.seed & 0xffffffffull);
  const dim3 tg((unsigned)((li.gen_tab + li.tile - 1) / li.tile), li.n_inst);
  cudaError_t e;
  if (db) {
    e = cudaFuncSetAttribute(general_tab_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
    if (e != cudaSuccess) return e;
    general_tab_kernel<true><<<tg, li.tile * GL, smem_bytes, s>>>(d_inst, li, arena, GL, garena);
  } else {
    e = cudaFuncSetAttribute(general_tab_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
    if (e != cudaSuccess) return e;
    general_tab_kernel<false><<<tg, li.tile * GL, smem_bytes, s>>>(d_inst, li, arena, GL, garena);
  }
  return cudaGetLastError();
}

int general_smem_bytes(int arena, int D, int T, int GL, bool db, bool glob) {
  int w4 = (D + 3) / 4;
  if ((w4 & 1) == 0) ++w4;
  return (glob ? 0 : arena * gen_row_stride(T, GL) * 4 * (db ? 2 : 1)) + T * 4 * w4;
}

// Scratch of the global-table mode: one [arena][row stride] slice (two with
// d/dbeta) per CTA of the contraction and of the tables kernel.
size_t general_scratch_floats(const LaunchInfo& li, int arena, int GL, bool db) {
  const size_t per = (size_t)arena * gen_row_stride(li.tile, GL) * (db ? 2 : 1);
  size_t ctas = (size_t)li.tile_begin[li.n_inst];
  if (li.gen_tab > 0) ctas = std::max(ctas, (size_t)((li.gen_tab + li.tile - 1) / li.tile) * li.n_inst);
  return per * ctas;
}

cudaError_t launch_general(const InstDev* d_inst, const LaunchInfo& li, int smem_bytes, int GL,
                           const int8_t* spins, double* logZR, double* dbeta, float* garena,
                           cudaStream_t s) {
  const int nblk = li.tile_begin[li.n_inst];
  if (nblk == 0) return cudaSuccess;
  // li.seed carries the arena size (floats) for this launch
  const int arena = (int)(li.seed & 0xffffffffull);
  const bool few = nblk <= GEN_FEW;
  auto kern = dbeta ? (few ? general_kernel<true, GEN_U> : general_kernel<true, 1>)
                    : (few ? general_kernel<false, GEN_U> : general_kernel<false, 1>);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  kern<<<nblk, li.tile * GL, smem_bytes, s>>>(d_inst, li, arena, GL, spins, logZR, dbeta, garena);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Magnetisation moments of the elimination components (observables from
// samples, Sec. 3).  The forward program run in the moment form: every table
// entry carries, besides its weight, the conditional mean and variance of the
// magnetisation of the spins already summed into it given its scope.  A
// step's product term at (x, sigma) has mean sigma + sum of its inputs' means
// and variance the sum of their variances (the inputs cover disjoint
// eliminated spins, independent given the scope), and summing sigma out
// merges the two terms (moment_mix).  A component's final entry gives the
// conditional mean and variance of its magnetisation; components are
// independent given the width set.  Tabulated components run their programs
// here too.  Tables: weights, means, variances, each [entry][sample].
// ---------------------------------------------------------------------------
__device__ __forceinline__ void run_component_mom(const GenDev& G, int c, const int8_t* s, float* A, float* Mu,
                                                  float* Q, int RS, int lane, int GL, float beta, double& mean,
                                                  double& var) {
  const int* H = G.fprog + G.fhdr[c];
  const int nsteps = H[0], fin = H[1];
  const int g0 = G.comp_step0[c];
  for (int st = 0; st < nsteps; ++st) {
    const StepRec r = step_at(G, g0 + st);
    const float h = field_of(G, r.fb, r.fc, s);
    const float ah = fabsf(h);
    const float fv[2] = {expf(beta * (h - ah)), expf(beta * (-h - ah))};
    const int M = 1 << r.m, E = 2 * M;
    const float* pp = G.pp + r.ppo;
    const unsigned short* mp = G.map + r.mo;
    const int out = r.out_live;
    float mx = 0.f;
    for (int x = lane; x < M; x += GL) {
      float tv[2], tm[2], tq[2];
#pragma unroll
      for (int sg = 0; sg < 2; ++sg) {
        const int ext = x | (sg << r.m);
        float p = fv[sg] * pp[ext], m = sg ? -1.f : 1.f, q = 0.f;
        for (int i = 0; i < r.nin; ++i) {
          const int a = (r.io[3 * i] + mp[i * E + ext]) * RS;
          p *= A[a];
          m += Mu[a];
          q += Q[a];
        }
        tv[sg] = p;
        tm[sg] = m;
        tq[sg] = q;
      }
      float v, m, q;
      moment_mix(tv[0], tm[0], tq[0], tv[1], tm[1], tq[1], v, m, q);
      A[(out + x) * RS] = v;
      Mu[(out + x) * RS] = m;
      Q[(out + x) * RS] = q;
      mx = fmaxf(mx, v);
    }
    mx = group_max(mx, GL);
    const float sc = pow2i(-exponent_of(mx));
    for (int x = lane; x < M; x += GL) A[(out + x) * RS] *= sc;
    __syncwarp();
  }
  if (lane == 0) {
    mean += (double)Mu[fin * RS];
    var += (double)Q[fin * RS];
  }
}

__global__ void __launch_bounds__(128) general_mom_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
                                                          int arena_floats, int GL, const int8_t* __restrict__ spins,
                                                          double* __restrict__ mag_mean, double* __restrict__ mag_var,
                                                          float* __restrict__ garena) {
  extern __shared__ float sm[];
  const int k = find_inst(li, blockIdx.x);
  const InstDev& I = inst[k];
  if (I.kind != 2) return;
  const int S = li.tile, slot = threadIdx.x / GL, lane = threadIdx.x % GL;
  const int b0 = (blockIdx.x - li.tile_begin[k]) * S, b = b0 + slot;
  const float beta = (float)li.beta[k];
  const int D = I.D, Dp = padded_bytes(D);
  const int RS = gen_row_stride(S, GL);
  const size_t cta_floats = (size_t)arena_floats * RS * 3;
  float* base = garena ? garena + (size_t)blockIdx.x * cta_floats : sm;
  float* A = base + slot;
  float* Mu = A + (size_t)arena_floats * RS;
  float* Q = Mu + (size_t)arena_floats * RS;
  int8_t* ssp = reinterpret_cast<int8_t*>(garena ? sm : sm + cta_floats);
  const GenDev& G = I.gen;
  const int n_valid = min(S, li.batch - b0);
  stage_spins(ssp, spins + I.spin_units * li.batch + (long long)b0 * D, n_valid, S, D, Dp);
  __syncthreads();
  const int8_t* s = ssp + slot * Dp;
  double mean = 0.0, var = 0.0;
  for (int c = 0; c < G.n_comp; ++c) run_component_mom(G, c, s, A, Mu, Q, RS, lane, GL, beta, mean, var);
  if (lane != 0 || b >= li.batch) return;
  int mw = 0;
  for (int j = 0; j < D; ++j) mw += s[j];
  const long long o = (long long)k * li.batch + b;
  mag_mean[o] = (double)mw + mean;
  mag_var[o] = var;
}

int general_mom_smem_bytes(int arena, int D, int T, int GL, bool glob) {
  int w4 = (D + 3) / 4;
  if ((w4 & 1) == 0) ++w4;
  return (glob ? 0 : arena * gen_row_stride(T, GL) * 4 * 3) + T * 4 * w4;
}

size_t general_mom_scratch_floats(const LaunchInfo& li, int arena, int GL) {
  return (size_t)arena * gen_row_stride(li.tile, GL) * 3 * (size_t)li.tile_begin[li.n_inst];
}

cudaError_t launch_general_mom(const InstDev* d_inst, const LaunchInfo& li, int smem_bytes, int arena, int GL,
                               const int8_t* spins, double* mag_mean, double* mag_var, float* garena,
                               cudaStream_t s) {
  const int nblk = li.tile_begin[li.n_inst];
  if (nblk == 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(general_mom_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  general_mom_kernel<<<nblk, li.tile * GL, smem_bytes, s>>>(d_inst, li, arena, GL, spins, mag_mean, mag_var, garena);
  return cudaGetLastError();
}

}  // namespace tnvan
