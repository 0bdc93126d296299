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
  b.pk = F[0] | (nin << 8);
  b.ppo = F[5];
  b.mo = F[6];
  b.out = F[7 + COL];
  b.in0 = nin > 0 ? F[9 + COL] : 0;
  b.in1 = nin > 1 ? F[12 + COL] : 0;
  b.in2 = nin > 2 ? F[15 + COL] : 0;
  b.h = 0.f;
  return b;
}
// The same read by each lane for itself: with one or two lanes a sample, and many
// CTAs to hide the reads, cheaper than the shuffles (65,536 samples, log Z_R and
// d/dbeta: n = 1,000 of width 2 985 and 1,439 us with shuffles, 926 and 1,263
// here; with four lanes, 32,768 samples of width 4, 1,088 and 1,567 against 1,190
// and 1,522).
template <int COL>
__device__ __forceinline__ Step read_step(const GenDev& G, int g, const int8_t* s) {
  Step r;
  r.f = G.fstep[g];
  const int* F = G.fprog + r.f;
  r.m = F[0];
  r.nin = F[3];
  r.ppo = F[5];
  r.mo = F[6];
  r.out = F[7 + COL];
  r.in[0] = r.nin > 0 ? F[9 + COL] : 0;
  r.in[1] = r.nin > 1 ? F[12 + COL] : 0;
  r.in[2] = r.nin > 2 ? F[15 + COL] : 0;
  r.h = field_of(G, F[1], F[2], s);
  return r;
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
  r.nin = pk >> 8;
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
// Launches of more CTAs than this (all that the dispatch sends here by itself;
// a capture that finds no buffers for the level kernels brings small ones too)
// take one entry at a time in half of the registers instead: there the CTAs in
// flight hide the latency, and the batch's dropped entries are only instructions
// (n = 500 of degree 3, width 4, with d/dbeta: 32,768 samples in 1,024 CTAs 1,068
// us four at a time, 653 one at a time; 4,096 samples in 256 CTAs 434 us four at
// a time, 526 one at a time).
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
template <bool DB, int U0, bool DIRECT>
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
    if (!DIRECT && j == 0) blk = load_block<0>(G, g0 + min(st + lane, nsteps - 1), s);
    const Step r = DIRECT ? read_step<0>(G, g0 + st, s) : block_step(blk, j, GL);
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
template <bool DB, int U0, bool DIRECT>
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
      run_component<DB, U0, DIRECT>(G, c, s, A, dA, RS, lane, GL, beta, lz, dl);
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
// Elimination by levels, lane = sample: 32 samples a CTA (tiles in turn), its
// warps take the tasks of one level after the other.  A table has one consumer,
// so the steps form a tree whose levels only need the level before: a plan of
// ~400 steps has ~30 levels (n = 500 of degree 3), and a step done by one warp
// needs no barrier inside (a lane only touches its own sample's column).  One
// step after the other, with any split of a step's entries, the chain of ~400
// steps' dependent reads and barriers set the time: 4,096 samples of that graph
// at width 8 take 193 us (338 with d/dbeta) by levels, 433 (717) step by step
// with the warps sharing a step's entries.  Every index is the same for a warp's
// lanes and every table access one 128-byte row.  A large step is cut into
// several tasks; their common scale follows after the level's barrier.  Tables
// of two neighbouring levels at a time are live (130 KB of shared memory for
// that graph).  What bounds it now: the levels' barriers (half of the stalls)
// and the plan's first reads from L2.  Each entry's arithmetic, and so every
// result, is that of step_table.
// ---------------------------------------------------------------------------
#define LV_U 4

// Scratch floats of a CTA of the level kernels.
__host__ __device__ __forceinline__ size_t general_levels_cta_floats(int live, int steps, bool db, int place) {
  return (size_t)steps * 64 + ((place & 1) ? 0 : (size_t)live * 32) + (db && !(place & 2) ? (size_t)live * 32 : 0);
}
__host__ __device__ __forceinline__ size_t general_levels_dJ_cta_floats(int total, int live, int gmax, int steps,
                                                                        int place) {
  return (size_t)steps * 64 + ((place & 1) ? 0 : (size_t)gmax * 32) + ((place & 2) ? 0 : (size_t)live * 32) +
         ((place & 4) ? 0 : (size_t)total * 32);
}

// A task's record, one int a lane; field i.
__device__ __forceinline__ int field(int rec, int i) { return __shfl_sync(0xffffffffu, rec, i); }

// The entries x0 .. x0 + nx - 1 of a step's table (in: the inputs' tables;
// nin >= 4: through lin), unscaled where nx > U or the step is cut.  Returns
// the largest.  fin: scale them here, by the returned maximum.
template <bool DB, int NIN, int U>
__device__ __forceinline__ float level_entries(const GenDev& G, int m, int nin, int ppo, int mo, int out, const int (&in)[3],
                                               const int* lin, int x0, int nx, const float (&fv)[2],
                                               const float (&fr)[2], float* A, float* dA, bool fin) {
  const int E = 2 << m, x1 = x0 + nx;
  const float* pp = G.pp + ppo;
  const float* pd = G.pp + G.n_pp + ppo;
  const unsigned short* mp = G.map + mo;
  float* oA = A + out * 32;
  float* oD = DB ? dA + out * 32 : nullptr;
  float av[U], dv[U], mx = 0.f;
  for (int xb = x0; xb < x1; xb += U) {
    float p[U][2], rr[U][2];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = min(xb + u, x1 - 1);
#pragma unroll
      for (int sg = 0; sg < 2; ++sg) {
        p[u][sg] = __ldg(pp + (x | (sg << m)));
        rr[u][sg] = DB ? __ldg(pd + (x | (sg << m))) : 0.f;
      }
    }
    if constexpr (NIN >= 0) {
      float val[NIN > 0 ? NIN : 1][U][2], dval[NIN > 0 ? NIN : 1][U][2];
#pragma unroll
      for (int i = 0; i < NIN; ++i)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int x = min(xb + u, x1 - 1);
#pragma unroll
          for (int sg = 0; sg < 2; ++sg) {
            const int q = (in[i] + __ldg(mp + i * E + (x | (sg << m)))) * 32;
            val[i][u][sg] = A[q];
            if (DB) dval[i][u][sg] = dA[q];
          }
        }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (DB && u >= nx) continue;  // no divisions for what is dropped
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
        const int x = min(xb + u, x1 - 1);
#pragma unroll
        for (int sg = 0; sg < 2; ++sg) {
          p[u][sg] = fv[sg] * p[u][sg];
          if (DB) rr[u][sg] = fr[sg] + rr[u][sg];
          for (int i = 0; i < nin; ++i) {
            const int q = (lin[2 * i] + mp[i * E + (x | (sg << m))]) * 32;
            const float v = A[q];
            p[u][sg] *= v;
            if (DB) rr[u][sg] += dA[q] / v;
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = xb + u;
      av[u] = __fadd_rn(p[u][0], p[u][1]);  // the products' own rounding: not contracted into the last one
      if (DB) dv[u] = fmaf(p[u][1], rr[u][1], p[u][0] * rr[u][0]);
      if (x >= x1) continue;
      mx = fmaxf(mx, av[u]);
      if (nx > U || !fin) {
        oA[x * 32] = av[u];
        if (DB) oD[x * 32] = dv[u];
      }
    }
  }
  if (!fin) return mx;
  const float sc = pow2i(-exponent_of(mx));
  if (nx <= U) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (u >= nx) continue;
      oA[(x0 + u) * 32] = av[u] * sc;
      if (DB) oD[(x0 + u) * 32] = dv[u] * sc;
    }
  } else {
#pragma unroll 4
    for (int x = x0; x < x1; ++x) {
      oA[x * 32] *= sc;
      if (DB) oD[x * 32] *= sc;
    }
  }
  return mx;
}

// A read that only brings its line into L1; landed() ends its wait.
__device__ __forceinline__ int touch(const void* p) {
  int v;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)3));
  return v;
}
__device__ __forceinline__ void landed(int v) { asm volatile("" ::"r"(v)); }
// Touch what the task of record rec reads first, a line a lane: bond products,
// maps, fields.  A plan's data is read once per tile, so without this every
// task starts with a chain of L2 reads.
template <bool DB>
__device__ __forceinline__ int touch_task(const GenDev& G, int rec, int lane) {
  const int w0 = field(rec, 0), m = w0 & 255, nin = w0 >> 9, M = 1 << m, x = field(rec, 6) + (lane & 1) * M;
  const int ppo = field(rec, 2), mo = field(rec, 3), fb = field(rec, 8), fc = field(rec, 9);
  const int j = lane >> 1;
  const void* p = nullptr;
  if (j == 0) p = G.pp + ppo + x;
  else if (j == 1) p = DB ? G.pp + G.n_pp + ppo + x : nullptr;
  else if (j == 2) p = fc == 0 ? nullptr : (lane & 1) ? static_cast<const void*>(G.fldJ + fb) : G.fld + 2 * fb;
  else if (j - 3 < nin && j < 9) p = G.map + mo + (j - 3) * 2 * M + x;
  return p ? touch(p) : 0;
}

// One level after the other, into A (and dA): FULL every table's own place,
// otherwise the level arena.  he[step]: this sample's field and the table's
// exponent.  red: the cut steps' maxima.  skip: leave out tabulated components.
// A, dA, he and red point at this lane's column.
template <bool DB, bool FULL>
__device__ __forceinline__ void level_sweep(const GenDev& G, const int8_t* s, float beta, float* A, float* dA,
                                            float2* he, float* red, bool skip, int wi, int NW, int lane) {
  const int t_end = G.n_lev > 0 ? G.llev[3 * G.n_lev - 1] : 0;
  auto record = [&](int t) {
    return t < t_end && lane < TNVAN_LTASK ? __ldg(G.ltask + (size_t)t * TNVAN_LTASK + lane) : 0;
  };
  int first = record(wi);
  for (int l = 0; l < G.n_lev; ++l) {
    const int t0 = G.llev[3 * l], tc = G.llev[3 * l + 1], t1 = G.llev[3 * l + 2];
    int nxt = first, far = record(t0 + wi + NW);
    first = record(t1 + wi);  // of the next level
    for (int t = t0 + wi; t < t1; t += NW) {
      const int rec = nxt;
      nxt = far;
      far = record(t + 2 * NW);
      const int tc0 = t + NW < t1 ? touch_task<DB>(G, nxt, lane) : 0;
      const int w0 = field(rec, 0), m = w0 & 255, nin = w0 >> 9;  // any number: the hub of a star has one per leaf
      if (skip && ((w0 >> 8) & 1)) continue;
      const int ppo = field(rec, 2), mo = field(rec, 3), out = field(rec, FULL ? 5 : 4);
      const int x0 = field(rec, 6), nx = field(rec, 7), slot = field(rec, 10);
      const int in[3] = {field(rec, FULL ? 17 : 14), field(rec, FULL ? 18 : 15), field(rec, FULL ? 19 : 16)};
      const float h = field_of(G, field(rec, 8), field(rec, 9), s), ah = fabsf(h);
      const float fv[2] = {expf(beta * (h - ah)), expf(beta * (-h - ah))};
      const float fr[2] = {h - ah, -h - ah};
      const int* lin = G.lin + field(rec, 13) + (FULL ? 1 : 0);
      const bool fin = slot < 0;
      float mx;
      constexpr int U3 = DB ? LV_U / 2 : LV_U;  // within 128 registers
      if (nx <= 2) {
        switch (nin) {
          case 0: mx = level_entries<DB, 0, 2>(G, m, nin, ppo, mo, out, in, lin, x0, nx, fv, fr, A, dA, fin); break;
          case 1: mx = level_entries<DB, 1, 2>(G, m, nin, ppo, mo, out, in, lin, x0, nx, fv, fr, A, dA, fin); break;
          case 2: mx = level_entries<DB, 2, 2>(G, m, nin, ppo, mo, out, in, lin, x0, nx, fv, fr, A, dA, fin); break;
          default: mx = level_entries<DB, -1, 2>(G, m, nin, ppo, mo, out, in, lin, x0, nx, fv, fr, A, dA, fin); break;
        }
      } else {
        switch (nin) {
          case 0: mx = level_entries<DB, 0, LV_U>(G, m, nin, ppo, mo, out, in, lin, x0, nx, fv, fr, A, dA, fin); break;
          case 1: mx = level_entries<DB, 1, LV_U>(G, m, nin, ppo, mo, out, in, lin, x0, nx, fv, fr, A, dA, fin); break;
          case 2: mx = level_entries<DB, 2, LV_U>(G, m, nin, ppo, mo, out, in, lin, x0, nx, fv, fr, A, dA, fin); break;
          case 3: mx = level_entries<DB, 3, U3>(G, m, nin, ppo, mo, out, in, lin, x0, nx, fv, fr, A, dA, fin); break;
          default: mx = level_entries<DB, -1, 2>(G, m, nin, ppo, mo, out, in, lin, x0, nx, fv, fr, A, dA, fin); break;
        }
      }
      const int step = field(rec, 1);
      if (fin) {
        he[step * 32] = make_float2(h, __int_as_float(exponent_of(mx)));
      } else {
        const int ch = field(rec, 11) >> 16;
        red[(slot + ch) * 32] = mx;
        if (ch == 0) he[step * 32].x = h;
      }
      landed(tc0);
    }
    landed(t1 + wi < t_end ? touch_task<DB>(G, first, lane) : 0);
    __syncthreads();
    if (tc == t0) continue;
    for (int t = t0 + wi; t < tc; t += NW) {  // the cut steps' scales
      const int rec = lane < TNVAN_LTASK ? __ldg(G.ltask + (size_t)t * TNVAN_LTASK + lane) : 0;
      if (skip && ((field(rec, 0) >> 8) & 1)) continue;
      const int out = field(rec, FULL ? 5 : 4), x0 = field(rec, 6), nx = field(rec, 7);
      const int slot = field(rec, 10), nch = field(rec, 11) & 0xffff, ch = field(rec, 11) >> 16, step = field(rec, 1);
      float mx = red[slot * 32];
      for (int j = 1; j < nch; ++j) mx = fmaxf(mx, red[(slot + j) * 32]);
      const int e = exponent_of(mx);
      const float sc = pow2i(-e);
      if (ch == 0) he[step * 32].y = __int_as_float(e);
#pragma unroll 4
      for (int x = x0; x < x0 + nx; ++x) {
        A[(out + x) * 32] *= sc;
        if (DB) dA[(out + x) * 32] *= sc;
      }
    }
    __syncthreads();
  }
}

// place: bit 0 A in shared memory, bit 1 dA too, else in this CTA's slice of
// gscr (as he always is).  tiles: li's CTAs, taken in turn by the launched ones.
template <bool DB>
__global__ void __launch_bounds__(512, 1) general_levels_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
                                                                int live, int steps, int red_slots, int place,
                                                                const int8_t* __restrict__ spins,
                                                                double* __restrict__ logZR, double* __restrict__ dbeta,
                                                                float* __restrict__ gscr) {
  extern __shared__ float sm[];
  __shared__ double term[16][32], dterm[DB ? 16 : 1][32];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, NW = blockDim.x >> 5;
  const size_t af = (size_t)live * 32;
  float* sp = sm;
  float* gp = gscr + (size_t)blockIdx.x * general_levels_cta_floats(live, steps, DB, place);
  float2* he = reinterpret_cast<float2*>(gp) + lane;
  gp += (size_t)steps * 64;
  float* A;
  float* dA = nullptr;
  if (place & 1) A = sp, sp += af;
  else A = gp, gp += af;
  if (DB) {
    if (place & 2) dA = sp, sp += af;
    else dA = gp;
    dA += lane;
  }
  A += lane;
  float* red = sp + lane;
  int8_t* ssp = reinterpret_cast<int8_t*>(sp + (size_t)red_slots * 32);
  for (int blk = blockIdx.x; blk < li.tile_begin[li.n_inst]; blk += gridDim.x) {
    const int k = find_inst(li, blk);
    const InstDev& I = inst[k];
    const GenDev& G = I.gen;
    const int b0 = (blk - li.tile_begin[k]) * 32, b = b0 + lane;
    const float beta = (float)li.beta[k];
    const int D = I.D, Dp = padded_bytes(D);
    stage_spins(ssp, spins + I.spin_units * li.batch + (long long)b0 * D, min(32, li.batch - b0), 32, D, Dp);
    __syncthreads();
    const int8_t* s = ssp + lane * Dp;
    const bool tab = li.gen_tab && G.n_tab > 0 && G.n_tab <= li.batch;  // tables built for this call
    if (!tab || G.n_tabc < G.n_comp) level_sweep<DB, false>(G, s, beta, A, dA, he, red, tab, wi, NW, lane);
    double lz = 0.0, dl = 0.0;
    for (int c0 = 0; c0 < G.n_comp; c0 += NW) {  // the components' terms, added up in their order
      const int c = c0 + wi;
      if (c < G.n_comp) {
        const int* cr = G.ctab + 5 * c;
        if (tab && cr[4] >= 0) {  // a tabulated component: one lookup
          const int x = boundary_index(G, cr, s);
          term[wi][lane] = G.tab_lz[cr[4] + x];
          if (DB) dterm[wi][lane] = G.tab_db[cr[4] + x];
        } else {
          const int g0 = G.comp_step0[c], g1 = G.comp_step0[c + 1], z0 = G.lroot[2 * c];
          int esum = 0;
          float hs = 0.f, hc = 0.f;  // as run_component
          for (int g = g0; g < g1; g += 8) {
            float2 q[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) q[j] = he[min(g + j, g1 - 1) * 32];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              if (g + j >= g1) break;
              const float y = fabsf(q[j].x) - hc;
              const float t2 = hs + y;
              hc = (t2 - hs) - y;
              hs = t2;
              esum += __float_as_int(q[j].y);
            }
          }
          const double hsum = (double)hs - (double)hc;
          const float z = A[z0 * 32];
          term[wi][lane] = (double)beta * hsum + (double)esum * 0.69314718055994530942 + (double)logf(z);
          if (DB) dterm[wi][lane] = hsum + (double)(dA[z0 * 32] / z);
        }
      }
      __syncthreads();
      if (wi == 0)
        for (int j = 0; j < min(NW, G.n_comp - c0); ++j) {
          lz += term[j][lane];
          if (DB) dl += dterm[j][lane];
        }
      __syncthreads();
    }
    if (wi == 0 && b < li.batch) {
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
    __syncthreads();  // spins free for the next tile
  }
}

// The tables of the tabulated components (at most TNVAN_TAB_MAX_K width-set
// neighbours): group g of instance k takes entry g of the concatenated
// tables, i.e. one component c and one boundary configuration x, sets the
// boundary spins of a spin row from the bits of x (the other spins do not
// enter c) and runs c's program alone, so that tab_lz[toff_c + x] = log Z_c
// and tab_db[..] its beta-derivative.  Built per call (they depend on beta)
// when they are smaller than the batch.
template <bool DB, bool DIRECT>
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
    run_component<DB, DIRECT ? 1 : GEN_U, DIRECT>(G, want, s, A, dA, RS, lane, GL, beta, lz, dl);
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
// The reverse sweep by levels (see general_levels_kernel): a forward sweep keeps
// every table, then from the last level back the g values of a level's steps,
// and after a barrier its bonds and its inputs' adjoints, each a warp's task.
// general_dJ_kernel's order of every FP32 sum is kept, so a group's row has the
// same bits in both forms (the rows are then added up in FP64, here by slices,
// there one after the other: d/dJ agrees to 1e-15): a bond's sum over a step's
// entries is made of W (that kernel's lanes per sample: 2, 4 or 8) chains x = w,
// w + W, ..., each added over the 32 / W samples of a group, then over the chains
// by the same tree, into the group's row; levels_dJ_reduce_kernel adds four
// groups' rows in turn, as that kernel's CTA did.  An edge has one bond in the
// plan, so rows are written, not added to.
// ---------------------------------------------------------------------------

// g of the extended indices of entries x0 .. x0 + nx - 1, into gb.
template <int NIN>
__device__ __forceinline__ void level_g(const GenDev& G, int m, int nin, int ppo, int mo, const int (&in)[3],
                                        const int* lin, int x0, int nx, const float (&fv)[2], const float* A,
                                        const float* Ab, float* gb, float scl) {
  constexpr int U = NIN >= 0 && NIN <= 2 ? 4 : 2;
  const int M = 1 << m, E = 2 * M, x1 = x0 + nx;
  const float* pp = G.pp + ppo;
  const unsigned short* mp = G.map + mo;
  for (int xb = x0; xb < x1; xb += U) {
    float p[U][2], ab[U], val[NIN > 0 ? NIN : 1][U][2];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = min(xb + u, x1 - 1);
      ab[u] = Ab[x * 32];
#pragma unroll
      for (int sg = 0; sg < 2; ++sg) {
        p[u][sg] = __ldg(pp + (x | (sg << m)));
#pragma unroll
        for (int i = 0; i < NIN; ++i) val[i][u][sg] = A[(in[i] + __ldg(mp + i * E + (x | (sg << m)))) * 32];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = xb + u;
      if (x >= x1) continue;
#pragma unroll
      for (int sg = 0; sg < 2; ++sg) {
        float v = fv[sg] * p[u][sg];
        if constexpr (NIN >= 0) {
#pragma unroll
          for (int i = 0; i < NIN; ++i) v *= val[i][u][sg];
        } else {
          for (int i = 0; i < nin; ++i) v *= A[(lin[2 * i] + mp[i * E + (x | (sg << m))]) * 32];
        }
        gb[(x | (sg << m)) * 32] = (ab[u] * scl) * v;
      }
    }
  }
}

// The adjoints of n entries of an input: each gathers the g of the R extended
// indices that read it, in index order (RR = R: four entries' loads at once).
template <int RR>
__device__ __forceinline__ void gather_g(const float* g, const unsigned short* inv, const float* av, float* ab, int n,
                                         int R) {
  if constexpr (RR > 0) {
    for (int e0 = 0; e0 < n; e0 += 4) {
      float a[4], v[4][RR];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = min(e0 + u, n - 1);
        a[u] = av[e * 32];
#pragma unroll
        for (int f = 0; f < RR; ++f) v[u][f] = g[__ldg(inv + e * RR + f) * 32];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (e0 + u >= n) continue;
        float sum = 0.f;
#pragma unroll
        for (int f = 0; f < RR; ++f) sum += v[u][f];
        ab[(e0 + u) * 32] = a[u] > 0.f ? 0.f + sum / a[u] : 0.f;
      }
    }
  } else {
#pragma unroll 2
    for (int e = 0; e < n; ++e) {
      const float a = av[e * 32];
      float sum = 0.f;
      for (int f = 0; f + 4 <= R; f += 4) {
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = g[__ldg(inv + e * R + f + j) * 32];
#pragma unroll
        for (int j = 0; j < 4; ++j) sum += v[j];
      }
      if (R < 4)
        for (int f = 0; f < R; ++f) sum += g[inv[e * R + f] * 32];
      ab[e * 32] = a > 0.f ? 0.f + sum / a : 0.f;
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
// The chains, times wscale (and sgn), added over the groups' samples and over the
// chains; to edge e of each group's row.
template <int W>
__device__ __forceinline__ void bond_store(const float (&v)[W], float wscale, float sgn, bool field_bond, float* rows,
                                           int stride, int e, int lane) {
  float u[W];
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const float q = wscale * v[w];
    u[w] = group_samples<W>(field_bond ? q * sgn : q);
  }
#pragma unroll
  for (int o = W / 2; o >= 1; o >>= 1)
#pragma unroll
    for (int w = 0; w < o; ++w) u[w] += u[w + o];
  if (e >= 0 && (lane & (32 / W - 1)) == 0) rows[(size_t)(lane / (32 / W)) * stride + e] = 0.f + u[0];
}

// place: bit 0 g values in shared memory, bit 1 the adjoints too, bit 2 the
// tables too, else in this CTA's slice of gscr.  rows of part: W per tile.
template <int W>
__global__ void __launch_bounds__(512, 1) general_levels_dJ_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
                                                                   int total, int live, int gmax, int steps,
                                                                   int red_slots, int place,
                                                                   const int8_t* __restrict__ spins,
                                                                   float* __restrict__ part, int part_stride,
                                                                   float* __restrict__ gscr) {
  extern __shared__ float sm[];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, NW = blockDim.x >> 5;
  float* sp = sm;
  float* gp = gscr + (size_t)blockIdx.x * general_levels_dJ_cta_floats(total, live, gmax, steps, place);
  float2* he = reinterpret_cast<float2*>(gp) + lane;
  gp += (size_t)steps * 64;
  auto take = [&](bool shared, int rows) {
    float*& q = shared ? sp : gp;
    float* r = q + lane;
    q += (size_t)rows * 32;
    return r;
  };
  float* gb = take(place & 1, gmax);
  float* Ab = take(place & 2, live);
  float* A = take(place & 4, total);
  float* red = take(true, red_slots);
  int8_t* ssp = reinterpret_cast<int8_t*>(sp);
  for (int blk = blockIdx.x; blk < li.tile_begin[li.n_inst]; blk += gridDim.x) {
    const int k = find_inst(li, blk);
    const InstDev& I = inst[k];
    const GenDev& G = I.gen;
    const int b0 = (blk - li.tile_begin[k]) * 32, b = b0 + lane;
    const float beta = (float)li.beta[k];
    const int D = I.D, Dp = padded_bytes(D);
    float* rows = part + (size_t)blk * W * part_stride;
    for (int e = threadIdx.x; e < W * part_stride; e += blockDim.x) rows[e] = 0.f;
    stage_spins(ssp, spins + I.spin_units * li.batch + (long long)b0 * D, min(32, li.batch - b0), 32, D, Dp);
    __syncthreads();
    const int8_t* s = ssp + lane * Dp;
    // per-sample weight of the bond sums (importance multipliers when given)
    const float wscale =
        b < li.batch ? beta / (float)li.batch * (li.wmul ? li.wmul[(long long)k * li.batch + b] : 1.f) : 0.f;
    level_sweep<false, true>(G, s, beta, A, nullptr, he, red, false, wi, NW, lane);
    for (int c = wi; c < G.n_comp; c += NW) Ab[G.lroot[2 * c] * 32] = 1.f / A[G.lroot[2 * c + 1] * 32];
    __syncthreads();
    auto level_first = [&](int l) {  // this warp's first task of level l
      const int t = l < 0 ? 0 : G.llev[3 * l] + wi;
      return l >= 0 && t < G.llev[3 * l + 2] && lane < TNVAN_LTASK ? __ldg(G.ltask + (size_t)t * TNVAN_LTASK + lane) : 0;
    };
    int first = level_first(G.n_lev - 1);
    for (int l = G.n_lev - 1; l >= 0; --l) {
      const int t0 = G.llev[3 * l], t1 = G.llev[3 * l + 2];
      auto record = [&](int t) {
        return t < t1 && lane < TNVAN_LTASK ? __ldg(G.ltask + (size_t)t * TNVAN_LTASK + lane) : 0;
      };
      int nxt = first, far = record(t0 + wi + NW);
      for (int t = t0 + wi; t < t1; t += NW) {
        const int rec = nxt;
        nxt = far;
        far = record(t + 2 * NW);
        const int tc0 = t + NW < t1 ? touch_task<false>(G, nxt, lane) : 0;
        const int w0 = field(rec, 0), m = w0 & 255, nin = w0 >> 9;
        const int ppo = field(rec, 2), mo = field(rec, 3), x0 = field(rec, 6), nx = field(rec, 7);
        const int in[3] = {field(rec, 17), field(rec, 18), field(rec, 19)};
        const int* lin = G.lin + field(rec, 13) + 1;
        const float2 q = he[field(rec, 1) * 32];
        const float h = q.x, ah = fabsf(h), scl = pow2i(-__float_as_int(q.y));
        const float fv[2] = {expf(beta * (h - ah)), expf(beta * (-h - ah))};
        const float* ab = Ab + field(rec, 4) * 32;
        float* g = gb + field(rec, 12) * 32;
        switch (nin) {
          case 0: level_g<0>(G, m, nin, ppo, mo, in, lin, x0, nx, fv, A, ab, g, scl); break;
          case 1: level_g<1>(G, m, nin, ppo, mo, in, lin, x0, nx, fv, A, ab, g, scl); break;
          case 2: level_g<2>(G, m, nin, ppo, mo, in, lin, x0, nx, fv, A, ab, g, scl); break;
          case 3: level_g<3>(G, m, nin, ppo, mo, in, lin, x0, nx, fv, A, ab, g, scl); break;
          default: level_g<-1>(G, m, nin, ppo, mo, in, lin, x0, nx, fv, A, ab, g, scl); break;
        }
        landed(tc0);
      }
      __syncthreads();
      const int u0 = G.blev[2 * l], u1 = G.blev[2 * l + 1];
      auto back = [&](int t) {
        return t < u1 && lane < TNVAN_BTASK ? __ldg(G.btask + (size_t)t * TNVAN_BTASK + lane) : 0;
      };
      int bnxt = back(u0 + wi);
      first = level_first(l - 1);
      for (int t = u0 + wi; t < u1; t += NW) {
        const int rec = bnxt;
        bnxt = back(t + NW);
        const int w0 = field(rec, 0), kind = w0 & 255, r1 = field(rec, 1), r3 = field(rec, 3), r4 = field(rec, 4);
        const float* g = gb + field(rec, 2) * 32;
        if (kind == 2) {  // input adjoints: each entry gathers the g of the extended indices that read it
          const int R = w0 >> 8, e0 = field(rec, 6);
          const unsigned short* inv = G.map + field(rec, 5);
          float* ab = Ab + (r3 + e0) * 32;
          const float* av = A + (r4 + e0) * 32;
          if (R == 2) gather_g<2>(g, inv, av, ab, r1, R);
          else if (R == 4) gather_g<4>(g, inv, av, ab, r1, R);
          else gather_g<0>(g, inv, av, ab, r1, R);
        } else {
          float v[W];
          bond_chains<W>(g, r1, kind == 0 ? -1 : r3, v);
          if (kind == 0) {
            for (int f = r3; f < r3 + r4; ++f)
              bond_store<W>(v, wscale, (float)s[G.fld[2 * f]], true, rows, part_stride, G.fld[2 * f + 1], lane);
          } else {
            bond_store<W>(v, wscale, 1.f, false, rows, part_stride, G.pairE[r4], lane);
          }
        }
      }
      landed(touch_task<false>(G, first, lane));
      __syncthreads();
    }
  }
}

// d/dJ from the group rows: 32 edges a CTA, 16 slices of the rows of four groups
// each, added in slice order.
template <int W>
__global__ void __launch_bounds__(512) levels_dJ_reduce_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
                                                               const float* __restrict__ part, int part_stride,
                                                               double* __restrict__ dJ) {
  __shared__ double acc[16][32];
  const int k = blockIdx.y;
  const InstDev& I = inst[k];
  const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
  if (I.kind != 2 || blockIdx.x * 32 >= I.n_edges) return;
  const int ng = (li.tile_begin[k + 1] - li.tile_begin[k]) * W, nr = (ng + 3) / 4;
  const float* p = part + (size_t)li.tile_begin[k] * W * part_stride + min(e, I.n_edges - 1);
  const int r0 = (int)((long long)nr * sl / 16), r1 = (int)((long long)nr * (sl + 1) / 16);
  double s = 0.0;
#pragma unroll 4
  for (int r = r0; r < r1; ++r) {
    float q[4], v = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) q[j] = 4 * r + j < ng ? p[(size_t)(4 * r + j) * part_stride] : 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) v += q[j];
    s += (double)v;
  }
  acc[sl][lane] = s;
  __syncthreads();
  if (sl != 0 || e >= I.n_edges) return;
  s = 0.0;
  for (int j = 0; j < 16; ++j) s += acc[j][lane];
  dJ[I.edge_off + e] += s;
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

// Shared memory sizes count in 64 bits: tables of a few 10^7 entries (a 12 x 1,024
// strip) pass 2^31 bytes, and a wrapped size would look as if they fitted.
static int clamp_bytes(long long b) { return (int)std::min<long long>(b, INT_MAX); }

// per-sample floats: 2 * arena + steps + gmax (tables, adjoints, scales, g)
int general_dJ_smem_bytes(int per_sample, int D, int n_edges, int T, int GL, bool glob) {
  int w4 = (D + 3) / 4;
  if ((w4 & 1) == 0) ++w4;
  return clamp_bytes((glob ? 0 : 4LL * per_sample * gen_row_stride(T, GL)) +
                     4LL * (T * GL / 32) * ((n_edges + 3) & ~3) + T * 4 * w4);
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

// Warps a CTA of the level kernels: a level's tasks, within 16; with more tiles
// than SMs half or a quarter of them in as many more CTAs an SM, where the
// shared memory allows it, so that one CTA's barriers are another's work.
static int levels_warps(int nblk, int tasks, int smem_bytes) {
  const int fit = 227 * 1024 / (smem_bytes + 10 * 1024);
  int w = tasks > 8 ? 16 : 8;
  while (w > 4 && nblk > 152 * (16 / w) && fit >= 2 * (16 / w)) w /= 2;
  return w;
}
// CTAs that fit the chip at once: 128 registers a thread and the shared memory.
static int levels_ctas(int nblk, int warps, int smem_bytes) {
  const int per_sm = std::max(1, std::min(16 / warps, 227 * 1024 / (smem_bytes + 10 * 1024)));
  return std::min(nblk, 152 * per_sm);
}
static int spin_bytes(int D) {
  int w4 = (D + 3) / 4;
  if ((w4 & 1) == 0) ++w4;
  return 32 * 4 * w4;
}
int general_levels_smem_bytes(int live, int red_slots, int D, bool db, int place) {
  const long long rows = ((place & 1) ? live : 0LL) + (db && (place & 2) ? live : 0) + red_slots;
  return clamp_bytes(128 * rows + spin_bytes(D));
}
size_t general_levels_scratch_floats(int live, int steps, bool db, int place, int nblk, int tasks, int smem_bytes) {
  return general_levels_cta_floats(live, steps, db, place) * levels_ctas(nblk, levels_warps(nblk, tasks, smem_bytes), smem_bytes);
}
cudaError_t launch_general_levels(const InstDev* d_inst, const LaunchInfo& li, int smem_bytes, int live, int steps,
                                  int red_slots, int tasks, int place, const int8_t* spins, double* logZR,
                                  double* dbeta, float* gscr, cudaStream_t s) {
  const int nblk = li.tile_begin[li.n_inst];
  if (nblk == 0) return cudaSuccess;
  auto kern = dbeta ? general_levels_kernel<true> : general_levels_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  const int nw = levels_warps(nblk, tasks, smem_bytes);
  kern<<<levels_ctas(nblk, nw, smem_bytes), 32 * nw, smem_bytes, s>>>(d_inst, li, live, steps, red_slots, place, spins,
                                                                    logZR, dbeta, gscr);
  return cudaGetLastError();
}
int general_levels_dJ_smem_bytes(int total, int live, int gmax, int red_slots, int D, int place) {
  const long long rows = ((place & 1) ? gmax : 0LL) + ((place & 2) ? live : 0) + ((place & 4) ? total : 0) + red_slots;
  return clamp_bytes(128 * rows + spin_bytes(D));
}
size_t general_levels_dJ_scratch_floats(int total, int live, int gmax, int steps, int place, int nblk, int tasks,
                                        int smem_bytes) {
  return general_levels_dJ_cta_floats(total, live, gmax, steps, place) *
         levels_ctas(nblk, levels_warps(nblk, tasks, smem_bytes), smem_bytes);
}
cudaError_t launch_general_levels_dJ(const InstDev* d_inst, const LaunchInfo& li, int smem_bytes, int W, int total,
                                     int live, int gmax, int steps, int red_slots, int tasks, int place, int max_edges,
                                     const int8_t* spins, float* part, int part_stride, double* dJ, float* gscr,
                                     cudaStream_t s) {
  const int nblk = li.tile_begin[li.n_inst];
  if (nblk == 0) return cudaSuccess;
  auto kern = W == 8 ? general_levels_dJ_kernel<8> : (W == 4 ? general_levels_dJ_kernel<4> : general_levels_dJ_kernel<2>);
  auto red = W == 8 ? levels_dJ_reduce_kernel<8> : (W == 4 ? levels_dJ_reduce_kernel<4> : levels_dJ_reduce_kernel<2>);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  const int nw = levels_warps(nblk, tasks, smem_bytes);
  kern<<<levels_ctas(nblk, nw, smem_bytes), 32 * nw, smem_bytes, s>>>(d_inst, li, total, live, gmax, steps, red_slots,
                                                                    place, spins, part, part_stride, gscr);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (max_edges == 0) return cudaSuccess;  // graphs without bonds
  red<<<dim3((max_edges + 31) / 32, li.n_inst), 512, 0, s>>>(d_inst, li, part, part_stride, dJ);
  return cudaGetLastError();
}

// The components' tables at this call's betas (li.gen_tab: the largest
// table; the contraction kernels then look them up).
cudaError_t launch_general_tables(const InstDev* d_inst, const LaunchInfo& li, int smem_bytes, bool db, int GL,
                                  float* garena, cudaStream_t s) {
  if (li.gen_tab <= 0) return cudaSuccess;
  const int arena = (int)(li.seed & 0xffffffffull);
  const dim3 tg((unsigned)((li.gen_tab + li.tile - 1) / li.tile), li.n_inst);
  const bool direct = GL <= 2;
  auto kern = db ? (direct ? general_tab_kernel<true, true> : general_tab_kernel<true, false>)
                 : (direct ? general_tab_kernel<false, true> : general_tab_kernel<false, false>);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  kern<<<tg, li.tile * GL, smem_bytes, s>>>(d_inst, li, arena, GL, garena);
  return cudaGetLastError();
}

int general_smem_bytes(int arena, int D, int T, int GL, bool db, bool glob) {
  int w4 = (D + 3) / 4;
  if ((w4 & 1) == 0) ++w4;
  return clamp_bytes((glob ? 0 : 4LL * arena * gen_row_stride(T, GL) * (db ? 2 : 1)) + T * 4 * w4);
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
  const bool few = nblk <= GEN_FEW, direct = GL <= 2;
  auto kern = dbeta ? (few ? general_kernel<true, GEN_U, false>
                           : (direct ? general_kernel<true, 1, true> : general_kernel<true, 1, false>))
                    : (few ? general_kernel<false, GEN_U, false>
                           : (direct ? general_kernel<false, 1, true> : general_kernel<false, 1, false>));
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
  return clamp_bytes((glob ? 0 : 12LL * arena * gen_row_stride(T, GL)) + T * 4 * w4);
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
