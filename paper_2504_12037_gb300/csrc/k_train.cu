// Reduction to F_q / log Z_IS (Eq. 9), the gradient's reduction over partial
// rows and the Adam update (Algorithm 1 step (d)).
#include <limits.h>
#include <math.h>

#include "common.cuh"

namespace tnvan {

// ---------------------------------------------------------------------------
// K7, two-pass FP64 form (the allocation-free entry point's reduction): per
// instance, over l_b = log Z_R(s_b) - log q(s_b).
// Pass 1 (grid n_part x n_inst): each CTA reduces a contiguous chunk to the
// mergeable tuple (n, mean, M2, max l, sum exp(l - max), #non-finite):
// Welford's update per sample, the pairwise update of Chan, Golub and
// LeVeque to merge (no shift taken from any one sample, so a non-finite
// first sample cannot spoil the sums).
// Pass 2 (grid n_inst): merges the n_part tuples in order and writes
//   stats[8k + 0..7] = F_q, F_IS, stderr, logZ_IS, mean l, #non-finite, var l, n;
// with no finite l_b every statistic is NaN and n = 0.
// Non-finite l_b are counted and left out.  FP64 throughout.
// ---------------------------------------------------------------------------
struct Tuple {
  double n, mean, M2, m, se, bad;
};

__device__ __forceinline__ Tuple merge(Tuple a, Tuple b) {
  if (a.n == 0.0) {
    b.bad += a.bad;
    return b;
  }
  if (b.n == 0.0) {
    a.bad += b.bad;
    return a;
  }
  Tuple r;
  r.n = a.n + b.n;
  const double d = b.mean - a.mean;
  r.mean = a.mean + d * (b.n / r.n);
  r.M2 = a.M2 + b.M2 + d * d * (a.n * b.n / r.n);
  r.bad = a.bad + b.bad;
  r.m = fmax(a.m, b.m);
  r.se = a.se * exp(a.m - r.m) + b.se * exp(b.m - r.m);
  return r;
}

__device__ __forceinline__ Tuple shfl_tuple(Tuple t, int o) {
  Tuple r;
  r.n = __shfl_xor_sync(0xffffffffu, t.n, o);
  r.mean = __shfl_xor_sync(0xffffffffu, t.mean, o);
  r.M2 = __shfl_xor_sync(0xffffffffu, t.M2, o);
  r.m = __shfl_xor_sync(0xffffffffu, t.m, o);
  r.se = __shfl_xor_sync(0xffffffffu, t.se, o);
  r.bad = __shfl_xor_sync(0xffffffffu, t.bad, o);
  return r;
}

__global__ void __launch_bounds__(256) reduce_part_kernel(const LaunchInfo li, int n_part,
                                                          const double* __restrict__ logZR,
                                                          const float* __restrict__ logq,
                                                          double* __restrict__ part) {
  const int k = blockIdx.y, p = blockIdx.x, B = li.batch;
  const long long base = (long long)k * B;
  const int chunk = (B + n_part - 1) / n_part;
  const int lo = p * chunk, hi = min(B, lo + chunk);
  Tuple acc = {0, 0, 0, 0, 0, 0};
  for (int b = lo + threadIdx.x; b < hi; b += blockDim.x) {
    const double l = logZR[base + b] - (double)logq[base + b];
    if (!isfinite(l)) {
      acc.bad += 1.0;
      continue;
    }
    acc.n += 1.0;
    const double d = l - acc.mean;
    acc.mean += d / acc.n;
    acc.M2 += d * (l - acc.mean);
    if (acc.n == 1.0) {
      acc.m = l;
      acc.se = 1.0;
    } else if (l > acc.m) {
      acc.se = acc.se * exp(acc.m - l) + 1.0;
      acc.m = l;
    } else {
      acc.se += exp(l - acc.m);
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc = merge(acc, shfl_tuple(acc, o));
  __shared__ Tuple red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    Tuple r = red[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) r = merge(r, red[w]);
    double* o = part + ((long long)k * n_part + p) * 6;
    o[0] = r.n;
    o[1] = r.mean;
    o[2] = r.M2;
    o[3] = r.m;
    o[4] = r.se;
    o[5] = r.bad;
  }
}

__global__ void reduce_final_kernel(const LaunchInfo li, int n_part, const double* __restrict__ part,
                                    double* __restrict__ stats) {
  const int k = blockIdx.x;
  if (threadIdx.x != 0) return;
  Tuple r = {0, 0, 0, 0, 0, 0};
  for (int p = 0; p < n_part; ++p) {
    const double* o = part + ((long long)k * n_part + p) * 6;
    Tuple t = {o[0], o[1], o[2], o[3], o[4], o[5]};
    r = merge(r, t);
  }
  double* s = stats + 8 * k;
  s[5] = r.bad;
  s[7] = r.n;
  if (r.n == 0.0) {  // no finite l_b: nothing to estimate
    const double nan = __longlong_as_double(0x7FF8000000000000ll);
    s[0] = s[1] = s[2] = s[3] = s[4] = s[6] = nan;
    return;
  }
  const double beta = li.beta[k];
  const double n = r.n;
  const double var = n > 1.0 ? r.M2 / (n - 1.0) : 0.0;
  const double lz = r.m + log(r.se) - log(n);
  s[0] = -r.mean / beta;
  s[1] = -lz / beta;
  s[2] = sqrt(var) / (beta * sqrt(n));
  s[3] = lz;
  s[4] = r.mean;
  s[6] = var;
}

// ---------------------------------------------------------------------------
// The same reduction in one launch (the context's form): the moment sums of
// l - K in float-float arithmetic -- each value an unevaluated sum hi + lo of
// two floats (error-free transforms: Knuth's TwoSum, Dekker's FastTwoSum, the
// FMA product error), about 48 significant bits, because FP64 is a narrow
// unit on this part -- and the logsumexp of the importance weights (log Z_IS)
// in FP64, about one FP64 exp per sample; the final statistics in FP64.
// Every CTA reduces its chunk and counts itself done on counters[k]; the
// last CTA of an instance merges the instance's n_part (<= 64) tuples with
// one warp -- a fixed tree over the chunk index, so the result does not
// depend on which CTA finishes last -- writes the statistics and re-arms the
// counter.
// ---------------------------------------------------------------------------
struct FF {
  float hi, lo;
};
__device__ __forceinline__ FF ff_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return FF{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ FF ff_fast_two_sum(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return FF{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ FF ff_add(FF x, FF y) {
  FF s = ff_two_sum(x.hi, y.hi);
  const FF t = ff_two_sum(x.lo, y.lo);
  s = ff_fast_two_sum(s.hi, __fadd_rn(s.lo, t.hi));
  return ff_fast_two_sum(s.hi, __fadd_rn(s.lo, t.lo));
}
__device__ __forceinline__ FF ff_mul(FF x, FF y) {
  const float p = __fmul_rn(x.hi, y.hi);
  float e = __fmaf_rn(x.hi, y.hi, -p);
  e = __fmaf_rn(x.hi, y.lo, e);
  e = __fmaf_rn(x.lo, y.hi, e);
  return ff_fast_two_sum(p, e);
}
__device__ __forceinline__ FF ff_neg(FF x) { return FF{-x.hi, -x.lo}; }
__device__ __forceinline__ bool ff_gt(FF a, FF b) { return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo); }
// double -> float-float with integer operations: hi = the top 24 significand
// bits (truncated, exact), lo = the next 29 bits rounded to a float.
__device__ __forceinline__ FF ff_from_double(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned sign = (unsigned)(u >> 63) << 31;
  const int E = (int)((u >> 52) & 0x7FFull);
  const int fe = E - 1023 + 127;
  if (E == 0x7FF) return FF{x != x ? __int_as_float(0x7FC00000) : __int_as_float((int)(sign | 0x7F800000u)), 0.f};
  if (fe <= 0 || fe >= 255) return FF{(float)x, 0.f};  // zero, tiny or huge: not met by log-likelihoods
  const unsigned long long M = u & 0xFFFFFFFFFFFFFull;
  const float hi = __int_as_float((int)(sign | ((unsigned)fe << 23) | (unsigned)(M >> 29)));
  const int le = E - 1075 + 127;  // 2^(E - 1023 - 52)
  const float lo = le > 0 ? __uint2float_rn((unsigned)(M & 0x1FFFFFFFull)) * __int_as_float(le << 23) : 0.f;
  return FF{hi, sign ? -lo : lo};
}
__device__ __forceinline__ double ff_to_double(FF x) { return (double)x.hi + (double)x.lo; }

// s1, s2: float-float sums of l - K and (l - K)^2; se: the sum of exp(l - e ln 2)
// in FP64, e an integer (m, once a chunk's sums are written) near its largest
// l / ln 2 (Eq. 9's log Z_IS is a logsumexp of the l_b, kept in FP64
// throughout); far: the sum of exp(l - m) instead, m the chunk's largest l.
struct TupleFF {
  int n, bad;
  FF s1, s2;
  double m, se;
  int far;
};
__device__ __forceinline__ FF shfl_ff(FF x, int o) {
  return FF{__shfl_xor_sync(0xffffffffu, x.hi, o), __shfl_xor_sync(0xffffffffu, x.lo, o)};
}
// partial tuples in a 6-double slot: n, bad, s1, s2 in words 0..5, m and se
// in doubles 3 and 4, far in word 10
__device__ __forceinline__ void st_tuple_ff(double* slot, const TupleFF& t) {
  float* f = reinterpret_cast<float*>(slot);
  reinterpret_cast<int*>(f)[0] = t.n;
  reinterpret_cast<int*>(f)[1] = t.bad;
  f[2] = t.s1.hi, f[3] = t.s1.lo, f[4] = t.s2.hi, f[5] = t.s2.lo;
  slot[3] = t.m;
  slot[4] = t.se;
  reinterpret_cast<int*>(f)[10] = t.far;
}
__device__ __forceinline__ TupleFF ld_tuple_ff(const double* slot) {
  const float* f = reinterpret_cast<const float*>(slot);
  const int* q = reinterpret_cast<const int*>(slot);
  return TupleFF{__ldcg(q), __ldcg(q + 1), FF{__ldcg(f + 2), __ldcg(f + 3)}, FF{__ldcg(f + 4), __ldcg(f + 5)},
                 __ldcg(slot + 3), __ldcg(slot + 4), __ldcg(q + 10)};
}
// Floats as integers of the same order (and back).
__device__ __forceinline__ int ordered(float f) {
  const int i = __float_as_int(f);
  return i ^ ((i >> 31) & 0x7FFFFFFF);
}
__device__ __forceinline__ float from_ordered(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7FFFFFFF)); }

// Sums of two lanes' tuples against the same maximum.
__device__ __forceinline__ void add_lane(TupleFF& r, int o) {
  r.n += __shfl_xor_sync(0xffffffffu, r.n, o);
  r.bad += __shfl_xor_sync(0xffffffffu, r.bad, o);
  r.s1 = ff_add(r.s1, shfl_ff(r.s1, o));
  r.s2 = ff_add(r.s2, shfl_ff(r.s2, o));
  r.se += __shfl_xor_sync(0xffffffffu, r.se, o);
}

// ln 2 times an integer, the exponent of the exponentials' common scale
// (formed the same way wherever a scale is taken off again).
__device__ __forceinline__ double scale_log(int e) { return (double)e * 0.69314718055994530942; }

// Each CTA (64 to 256 threads) reduces a chunk in two passes over its samples:
// the chunk's largest l first (in FP32: it only picks a power of two 2^e near
// exp(max l)), then per sample one FP64 exp(l - e ln 2) and the float-float
// moment sums, merged over lanes and warps by a fixed tree.  The last CTA of an
// instance takes the n_part (<= 64) chunk sums to the largest e -- an exact
// power of two each -- and adds them in a fixed tree, so the result does not
// depend on which CTA finishes last.  Bound by a chain of latencies (loads, one
// exp, about ten float-float additions, the hand-over between CTAs, one log):
// FP64 is a narrow unit on this part, so small batches are spread over CTAs of
// 64 samples, maxima are integer warp reductions, chunks are rescaled without
// exponentials, and what depends on the batch size alone (its log, reciprocals)
// comes from the host.  1,024 samples: 14.8 us with FP64 maxima, an exp per
// chunk and one thread merging the warps, 11 us here (3 x 4,096: 15.1 and
// 11).  A chunk whose largest l lies where FP32 no longer places it within the
// exponentials' range (|l| > RED_FAR: its spacing there is 64) takes the FP64
// maximum as its scale, and an instance with such a chunk rescales by
// exponentials.
#define RED_FAR 6e8f
struct BatchConsts {  // of n samples: 1 / n, 1 / (n - 1) (0 for n = 1), ln n, 1 / sqrt n
  double inv_n, inv_n1, ln_n, rsqrt_n;
};
__global__ void __launch_bounds__(256) reduce_kernel(const LaunchInfo li, int n_part, const BatchConsts bc,
                                                     const double* __restrict__ logZR,
                                                     const float* __restrict__ logq, double* __restrict__ part,
                                                     double* __restrict__ stats, int* __restrict__ counters,
                                                     int k0) {
  const int k = blockIdx.y + k0, p = blockIdx.x, B = li.batch;
  const long long base = (long long)k * B;
  // the shift of the moment sums: l_0 when finite (else 0)
  FF K = ff_add(ff_from_double(logZR[base]), FF{-logq[base], 0.f});
  if (!isfinite(K.hi) || !isfinite(K.lo)) K = FF{0.f, 0.f};
  const FF negK = ff_neg(K);
  const int chunk = (B + n_part - 1) / n_part;
  const int lo = p * chunk, hi = min(B, lo + chunk);
  const int l = threadIdx.x & 31, nw = blockDim.x >> 5;
  __shared__ int redi[8];
  __shared__ double redd[8];
  __shared__ TupleFF red[8];
  __shared__ int last;
  // pass 1: the chunk's largest finite l
  float mf = -INFINITY;
  for (int b = lo + threadIdx.x; b < hi; b += blockDim.x) {
    const double ld = logZR[base + b] - (double)logq[base + b];
    if (isfinite(ld)) mf = fmaxf(mf, (float)ld);
  }
  int mi = __reduce_max_sync(0xffffffffu, ordered(mf));
  if (l == 0) redi[threadIdx.x >> 5] = mi;
  __syncthreads();
  mi = redi[0];
  for (int w = 1; w < nw; ++w) mi = max(mi, redi[w]);
  const float top = from_ordered(mi);
  const bool far = !(fabsf(top) <= RED_FAR);  // the same for the CTA; also no finite l
  const int e2 = far ? 0 : (int)ceilf(top * 1.44269504f);
  double mx = scale_log(e2);
  if (far) {
    double md = -INFINITY;
    for (int b = lo + threadIdx.x; b < hi; b += blockDim.x) {
      const double ld = logZR[base + b] - (double)logq[base + b];
      if (isfinite(ld)) md = fmax(md, ld);
    }
    for (int o = 16; o > 0; o >>= 1) md = fmax(md, __shfl_xor_sync(0xffffffffu, md, o));
    if (l == 0) redd[threadIdx.x >> 5] = md;
    __syncthreads();
    mx = redd[0];
    for (int w = 1; w < nw; ++w) mx = fmax(mx, redd[w]);
    if (!isfinite(mx)) mx = 0.0;  // no finite l: any scale (the sums stay zero)
  }
  // pass 2: exp sums at that scale, moment sums, counts
  TupleFF acc = {0, 0, {0.f, 0.f}, {0.f, 0.f}, 0.0, 0.0, 0};
  for (int b = lo + threadIdx.x; b < hi; b += blockDim.x) {
    const double z = logZR[base + b];
    const float q = logq[base + b];
    const double ld = z - (double)q;
    if (!isfinite(ld)) {
      acc.bad += 1;
      continue;
    }
    const FF d = ff_add(ff_add(ff_from_double(z), FF{-q, 0.f}), negK);
    acc.s1 = ff_add(acc.s1, d);
    acc.s2 = ff_add(acc.s2, ff_mul(d, d));
    acc.se += exp(ld - mx);
    acc.n += 1;
  }
  for (int o = 16; o > 0; o >>= 1) add_lane(acc, o);
  if (l == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    TupleFF r = red[l < nw ? l : 0];
    if (l >= nw) r = TupleFF{0, 0, {0.f, 0.f}, {0.f, 0.f}, 0.0, 0.0, 0};
    for (int o = 4; o > 0; o >>= 1) add_lane(r, o);
    if (l == 0) {
      r.m = far ? mx : (double)e2;
      r.far = far;
      st_tuple_ff(part + ((long long)k * n_part + p) * 6, r);
      __threadfence();
      last = atomicAdd(counters + k, 1) == n_part - 1;
    }
  }
  __syncthreads();
  if (!last || threadIdx.x >= 32) return;
  const double inv_beta = 1.0 / li.beta[k];
  __threadfence();
  // the instance's chunks: lane l holds chunks l and l + 32
  TupleFF r = {0, 0, {0.f, 0.f}, {0.f, 0.f}, 0.0, 0.0, 0};
  TupleFF r2 = r;
  if (l < n_part) r = ld_tuple_ff(part + ((long long)k * n_part + l) * 6);
  if (l + 32 < n_part) r2 = ld_tuple_ff(part + ((long long)k * n_part + l + 32) * 6);
  double top_l;  // log of the sums' common scale
  if (!__any_sync(0xffffffffu, (r.n && r.far) || (r2.n && r2.far))) {
    const int ea = r.n ? (int)r.m : INT_MIN, eb = r2.n ? (int)r2.m : INT_MIN;
    const int E = __reduce_max_sync(0xffffffffu, max(ea, eb));
    top_l = scale_log(E);
    r.se = r.n ? scalbn(r.se, max(ea - E, -2000)) : 0.0;
    r2.se = r2.n ? scalbn(r2.se, max(eb - E, -2000)) : 0.0;
  } else {
    const double ma = r.far ? r.m : scale_log((int)r.m), mb = r2.far ? r2.m : scale_log((int)r2.m);
    top_l = fmax(r.n ? ma : -INFINITY, r2.n ? mb : -INFINITY);
    for (int o = 16; o > 0; o >>= 1) top_l = fmax(top_l, __shfl_xor_sync(0xffffffffu, top_l, o));
    r.se = r.n ? r.se * exp(ma - top_l) : 0.0;
    r2.se = r2.n ? r2.se * exp(mb - top_l) : 0.0;
  }
  if (n_part > 32) {
    r.se += r2.se;
    r.n += r2.n;
    r.bad += r2.bad;
    r.s1 = ff_add(r.s1, r2.s1);
    r.s2 = ff_add(r.s2, r2.s2);
  }
  for (int o = 16; o > 0; o >>= 1) add_lane(r, o);
  const int n_ = r.n, bad_ = r.bad;
  // FP64 statistics
  double inv_n = bc.inv_n, inv_n1 = bc.inv_n1, ln_n = bc.ln_n, rsqrt_n = bc.rsqrt_n;
  const double n = (double)n_;
  if (bad_) {  // some l_b left out
    inv_n = 1.0 / n;
    inv_n1 = n_ > 1 ? 1.0 / (n - 1.0) : 0.0;
    ln_n = log(n);
    rsqrt_n = 1.0 / sqrt(n);
  }
  const double s1d = ff_to_double(r.s1), s2d = ff_to_double(r.s2);
  const double mean_d = s1d * inv_n;
  const double var = fmax(s2d - s1d * mean_d, 0.0) * inv_n1;
  double f = l == 0 ? r.se : var;  // log of one lane's value, square root of the others'
  if (l == 0) f = log(f);
  else f = sqrt(f);
  const double sd = __shfl_sync(0xffffffffu, f, 1);
  if (l != 0) return;
  const double nan = __longlong_as_double(0x7FF8000000000000ll);
  const double mean = n_ ? ff_to_double(K) + mean_d : nan;
  const double lz = n_ ? top_l + f - ln_n : nan;
  double* st = stats + 8 * k;
  st[0] = -mean * inv_beta;
  st[1] = -lz * inv_beta;
  st[2] = sd * inv_beta * rsqrt_n;
  st[3] = lz;
  st[4] = mean;
  st[5] = (double)bad_;
  st[6] = var;
  st[7] = n;
  counters[k] = 0;
}

cudaError_t launch_reduce(const InstDev*, const LaunchInfo& li, const double* logZR,
                          const float* logq, double* stats, int* counters, cudaStream_t s, int k0, int k1) {
  if (k1 < 0) k1 = li.n_inst;
  if (k1 <= k0) return cudaSuccess;
  // chunks of >= 64 samples, at most 64 per instance; a thread per sample up to 256
  int n_part = (li.batch + 63) / 64;
  if (n_part > 64) n_part = 64;
  if (n_part < 1) n_part = 1;
  const int chunk = (li.batch + n_part - 1) / n_part;
  const int threads = chunk <= 64 ? 64 : (chunk <= 128 ? 128 : 256);
  // partial tuples live right after the stats block
  double* part = stats + 8 * TNVAN_MAX_INST;
  const double n = li.batch;
  const BatchConsts bc = {1.0 / n, n > 1.0 ? 1.0 / (n - 1.0) : 0.0, log(n), 1.0 / sqrt(n)};
  reduce_kernel<<<dim3(n_part, k1 - k0), threads, 0, s>>>(li, n_part, bc, logZR, logq, part, stats, counters, k0);
  return cudaGetLastError();
}

// Merge of Eq. 9 statistics rows computed on disjoint parts of one batch
// (data-parallel ranks), parts[(p * n_inst + k) * 8 + 0..7] in the layout of
// the reduction, into stats[8k + 0..7] for the union of the parts.  Each row
// is taken as the mergeable tuple (n, mean l, M2 = var (n - 1), log sum e^l =
// logZ_IS + ln n) and the parts are combined in index order by the pairwise
// update of Chan, Golub and LeVeque (1979) for the mean and M2 and a
// logaddexp for the log-sum; one thread per instance, so the result does not
// depend on the launch.  One part is copied unchanged.
__global__ void merge_stats_kernel(const LaunchInfo li, int n_parts, const double* __restrict__ parts,
                                   double* __restrict__ stats) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= li.n_inst) return;
  const double* p0 = parts + 8 * k;
  double* st = stats + 8 * k;
  if (n_parts == 1) {
    for (int j = 0; j < 8; ++j) st[j] = p0[j];
    return;
  }
  double n = 0.0, mean = 0.0, M2 = 0.0, lse = 0.0, bad = 0.0;
  for (int p = 0; p < n_parts; ++p) {
    const double* q = parts + ((long long)p * li.n_inst + k) * 8;
    const double nb = q[7];
    bad += q[5];
    if (!(nb > 0.0)) continue;
    const double mb = q[4], M2b = nb > 1.0 ? q[6] * (nb - 1.0) : 0.0, lb = q[3] + log(nb);
    if (n == 0.0) {
      n = nb, mean = mb, M2 = M2b, lse = lb;
      continue;
    }
    const double N = n + nb, d = mb - mean;
    mean += d * (nb / N);
    M2 += M2b + d * d * (n * nb / N);
    lse = fmax(lse, lb) + log1p(exp(-fabs(lse - lb)));
    n = N;
  }
  const double beta = li.beta[k];
  const double var = n > 1.0 ? M2 / (n - 1.0) : 0.0;
  const double lz = lse - log(n);
  st[0] = -mean / beta;
  st[1] = -lz / beta;
  st[2] = sqrt(var) / (beta * sqrt(n));
  st[3] = lz;
  st[4] = mean;
  st[5] = bad;
  st[6] = var;
  st[7] = n;
}

cudaError_t launch_merge_stats(const LaunchInfo& li, int n_parts, const double* parts, double* stats,
                               cudaStream_t s) {
  merge_stats_kernel<<<(li.n_inst + 127) / 128, 128, 0, s>>>(li, n_parts, parts, stats);
  return cudaGetLastError();
}

// Adam (Kingma & Ba 2015) on one entry, bias corrections bc1 = 1 - b1^t,
// bc2 = 1 - b2^t.  The one definition both Adam kernels use.
__device__ __forceinline__ void adam_entry(float& p, float& m, float& v, float g, const AdamArgs& a, float bc1,
                                           float bc2) {
  const float mi = a.b1 * m + (1.f - a.b1) * g;
  const float vi = a.b2 * v + (1.f - a.b2) * g * g;
  m = mi;
  v = vi;
  p -= a.lr * (mi / bc1) / (sqrtf(vi / bc2) + a.eps);
}

// The bias corrections of this launch: the host's, or (device step counter)
// formed by one thread of the CTA in FP64 (a narrow unit here) from
// t = t_base + *t_dev.
__device__ __forceinline__ void adam_corrections(const AdamArgs& a, float& bc1, float& bc2) {
  bc1 = a.bc1;
  bc2 = a.bc2;
  if (a.t_dev) {
    __shared__ float bc[2];
    if (threadIdx.x == 0) {
      const double t = (double)(a.t_base + (long long)*a.t_dev);
      bc[0] = (float)(1.0 - exp(t * log((double)a.b1)));
      bc[1] = (float)(1.0 - exp(t * log((double)a.b2)));
    }
    __syncthreads();
    bc1 = bc[0];
    bc2 = bc[1];
  }
}

// Sum the chunk partials of every instance (fixed order: deterministic) and
// scatter from the packed, degree-sorted layout to the caller's natural
// layout; entries outside the MADE masks get 0.  With ADAM the same thread
// then applies Adam to that entry of the instance's own parameters
// (tnvan_set_made's pointer) with the moments at the gradient's offset, so a
// training step needs no separate optimizer pass over the gradient.
template <bool ADAM>
__global__ void grad_reduce_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
                                   const float* __restrict__ partials, long long part_stride,
                                   float* __restrict__ grad, const AdamArgs adam, int k0) {
  const int k = blockIdx.y + k0;
  if ((li.skip[k >> 5] >> (k & 31)) & 1u) return;  // reduced by another backward form
  const MadeDev& md = inst[k].made;
  float bc1 = 1.f, bc2 = 1.f;
  if (ADAM) adam_corrections(adam, bc1, bc2);
  const int p0 = li.tile_begin[k], p1 = li.tile_begin[k + 1];
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < md.n_params;
       e += (long long)gridDim.x * blockDim.x) {
    // eight independent partial sums keep eight loads in flight; fixed order
    float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    int p = p0;
    for (; p + 8 <= p1; p += 8)
#pragma unroll
      for (int j = 0; j < 8; ++j) a[j] += partials[(long long)(p + j) * part_stride + e];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (p + j < p1) a[j] += partials[(long long)(p + j) * part_stride + e];
    const float s = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
    int r = (int)e;  // a network's parameter count fits in 32 bits (checked at set-up)
    long long nat = -1;
    float gv = s;
    for (int l = 0; l < md.n_layers; ++l) {
      const LayerDev& L = md.layer[l];
      const int nw = L.nout * L.nin;
      if (r < nw) {
        const int o = r / L.nin, i = r - o * L.nin;
        const int no = L.perm_out ? L.perm_out[o] : o;
        const int ni = L.perm_in ? L.perm_in[i] : i;
        const bool conn = L.strict ? (L.deg_out[o] > L.deg_in[i]) : (L.deg_out[o] >= L.deg_in[i]);
        nat = L.src_off + (long long)no * L.nin + ni;
        gv = conn ? s : 0.f;
        break;
      }
      r -= nw;
      if (r < L.nout) {
        nat = L.src_off + nw + (L.perm_out ? L.perm_out[r] : r);
        break;
      }
      r -= L.nout;
    }
    if (nat < 0) continue;
    const long long o = md.param_off + nat;
    grad[o] = gv;
    if (ADAM) adam_entry(md.raw[nat], adam.m[o], adam.v[o], gv, adam, bc1, bc2);
  }
}

cudaError_t launch_grad_reduce(const InstDev* d_inst, const LaunchInfo& li, const float* partials,
                               int part_stride, float* grad, cudaStream_t s, const AdamArgs* adam, int k0, int k1) {
  if (k1 < 0) k1 = li.n_inst;
  if (k1 <= k0) return cudaSuccess;
  // one parameter per thread (the row stride bounds every instance's count),
  // at most 256 CTAs per instance and about 4096 per launch (a launch over
  // many instances strides instead)
  const int cap = 4096 / (k1 - k0) > 16 ? 4096 / (k1 - k0) : 16;
  int gx = (int)((part_stride + 255) / 256);
  gx = gx < cap ? gx : cap;
  gx = gx < 256 ? gx : 256;
  const dim3 grid((unsigned)(gx > 1 ? gx : 1), k1 - k0);
  if (adam)
    grad_reduce_kernel<true><<<grid, 256, 0, s>>>(d_inst, li, partials, part_stride, grad, *adam, k0);
  else
    grad_reduce_kernel<false><<<grid, 256, 0, s>>>(d_inst, li, partials, part_stride, grad, AdamArgs{}, k0);
  return cudaGetLastError();
}

// Importance weights of tnvan_observables as multipliers B w_b =
// exp(l_b - logZ_IS), w_b = exp(l_b) / sum_b' exp(l_b') (self-normalised;
// logZ_IS = logsumexp_b l_b - ln B from the F_q reduction's statistics).
__global__ void obs_weights_kernel(const LaunchInfo li, const double* __restrict__ logZR,
                                   const float* __restrict__ logq, const double* __restrict__ stats,
                                   float* __restrict__ wmul) {
  const int k = blockIdx.y;
  const double lz = stats[8 * k + 3];
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < li.batch; b += gridDim.x * blockDim.x) {
    const long long o = (long long)k * li.batch + b;
    wmul[o] = (float)exp(logZR[o] - (double)logq[o] - lz);
  }
}

// Per instance (one CTA each): sum_b m_b E_b, sum_b E_b and sum_b m_b^2 with
// E_b = -dbeta_b and m_b the multipliers above, in a fixed order (FP64).
__global__ void obs_energy_kernel(const LaunchInfo li, const double* __restrict__ dbeta,
                                  const float* __restrict__ wmul, double* __restrict__ out) {
  const int k = blockIdx.x;
  double a = 0.0, e = 0.0, q = 0.0;
  for (int b = threadIdx.x; b < li.batch; b += blockDim.x) {
    const long long o = (long long)k * li.batch + b;
    const double E = -dbeta[o], m = (double)wmul[o];
    a += m * E;
    e += E;
    q += m * m;
  }
  __shared__ double red[3][256];
  red[0][threadIdx.x] = a;
  red[1][threadIdx.x] = e;
  red[2][threadIdx.x] = q;
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h)
      for (int j = 0; j < 3; ++j) red[j][threadIdx.x] += red[j][threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double B = (double)li.batch;
    out[3 * k + 0] = red[0][0] / B;      // U  = sum_b w_b E_b
    out[3 * k + 1] = red[1][0] / B;      // U_q = mean_b E_b
    out[3 * k + 2] = B * B / red[2][0];  // effective sample size 1 / sum_b w_b^2
  }
}

cudaError_t launch_observables(const LaunchInfo& li, const double* logZR, const float* logq, const double* stats,
                               const double* dbeta, float* wmul, double* out, bool energies, cudaStream_t s) {
  if (li.n_inst == 0 || li.batch == 0) return cudaSuccess;
  if (!energies) {
    obs_weights_kernel<<<dim3(32, li.n_inst), 256, 0, s>>>(li, logZR, logq, stats, wmul);
    return cudaGetLastError();
  }
  obs_energy_kernel<<<li.n_inst, 256, 0, s>>>(li, dbeta, wmul, out);
  return cudaGetLastError();
}

// Per instance (one CTA each), in a fixed order (FP64), with m_b the
// multipliers B w_b above, mu_b = E[M | s_b] and v_b = Var(M | s_b):
//   out[5k+0] = sum_b m_b mu_b / B                 (<M>, importance-weighted)
//   out[5k+1] = sum_b m_b (mu_b^2 + v_b) / B       (<M^2>)
//   out[5k+2] = mean_b mu_b,  out[5k+3] = mean_b (mu_b^2 + v_b)   (the same under q)
//   out[5k+4] = B^2 / sum_b m_b^2                  (effective sample size)
__global__ void obs_mag_kernel(const LaunchInfo li, const double* __restrict__ mean, const double* __restrict__ var,
                               const float* __restrict__ wmul, double* __restrict__ out) {
  const int k = blockIdx.x;
  double a[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int b = threadIdx.x; b < li.batch; b += blockDim.x) {
    const long long o = (long long)k * li.batch + b;
    const double mu = mean[o], m2 = mu * mu + var[o], w = (double)wmul[o];
    a[0] += w * mu;
    a[1] += w * m2;
    a[2] += mu;
    a[3] += m2;
    a[4] += w * w;
  }
  __shared__ double red[5][256];
  for (int j = 0; j < 5; ++j) red[j][threadIdx.x] = a[j];
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h)
      for (int j = 0; j < 5; ++j) red[j][threadIdx.x] += red[j][threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double B = (double)li.batch;
    for (int j = 0; j < 4; ++j) out[5 * k + j] = red[j][0] / B;
    out[5 * k + 4] = B * B / red[4][0];
  }
}

cudaError_t launch_obs_mag(const LaunchInfo& li, const double* mean, const double* var, const float* wmul,
                           double* out, cudaStream_t s) {
  if (li.n_inst == 0 || li.batch == 0) return cudaSuccess;
  obs_mag_kernel<<<li.n_inst, 256, 0, s>>>(li, mean, var, wmul, out);
  return cudaGetLastError();
}

// REINFORCE weights w_b = -(l_b - mean_b l) / (beta B) per instance (Eq. 10
// with the batch-mean baseline), FP32 copy for the tensor-core backward.
// Eq. 10's per-sample weights w[k][b]; with s16, also the spins of every
// instance not marked in li.skip as BF16 rows of D rounded up to 8 (zeros
// beyond D), instance k at sum_{j<k} batch * r8(D_j): the GEMM chain's spin
// operands.
__global__ void reinforce_w_kernel(const InstDev* __restrict__ inst, const LaunchInfo li,
                                   const double* __restrict__ logZR, const float* __restrict__ logq,
                                   const double* __restrict__ stats, float* __restrict__ w,
                                   const int8_t* __restrict__ spins, uint16_t* __restrict__ s16) {
  const int k = blockIdx.y;
  const double mean = stats[8 * k + 4];
  const double sc = -1.0 / (li.beta[k] * stats_batch(stats + 8 * k));
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < li.batch; b += gridDim.x * blockDim.x) {
    const long long o = (long long)k * li.batch + b;
    w[o] = (float)(sc * (logZR[o] - (double)logq[o] - mean));
  }
  if (!s16 || ((li.skip[k >> 5] >> (k & 31)) & 1u)) return;  // skipped: another backward form reads the spins
  long long off = 0;
  for (int j = 0; j < k; ++j) off += (long long)li.batch * ((inst[j].D + 7) & ~7);
  const int D = inst[k].D, G8 = (D + 7) >> 3;  // 8-spin groups per row
  const int8_t* src = spins + inst[k].spin_units * li.batch;
  const long long n = (long long)li.batch * G8;
  uint4* dst = reinterpret_cast<uint4*>(s16 + off);  // 16-byte aligned: off is a multiple of 8
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const long long b = e / G8;
    const int i0 = (int)(e - b * G8) * 8;
    uint32_t h[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t v = 0;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int i = i0 + 2 * q + j;
        const uint32_t x = i < D ? (src[b * D + i] > 0 ? 0x3F80u : 0xBF80u) : 0u;
        v |= x << (16 * j);
      }
      h[q] = v;
    }
    dst[e] = make_uint4(h[0], h[1], h[2], h[3]);
  }
}

cudaError_t launch_reinforce_w(const InstDev* d_inst, const LaunchInfo& li, const double* logZR, const float* logq,
                               const double* stats, float* w, const int8_t* spins, uint16_t* s16, cudaStream_t s) {
  if (li.n_inst == 0 || li.batch == 0) return cudaSuccess;
  reinforce_w_kernel<<<dim3(32, li.n_inst), 256, 0, s>>>(d_inst, li, logZR, logq, stats, w, spins, s16);
  return cudaGetLastError();
}

// Adam over a flat array (tnvan_adam).  With t_dev, the step is
// t_base + *t_dev (a device step counter, for replayed CUDA graphs).
__global__ void adam_kernel(long long n, float* __restrict__ p, const float* __restrict__ g, const AdamArgs a) {
  float bc1, bc2;
  adam_corrections(a, bc1, bc2);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    adam_entry(p[i], a.m[i], a.v[i], g[i], a, bc1, bc2);
}

cudaError_t launch_adam(long long n, float* p, const float* g, const AdamArgs& a, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  long long nb = (n + 255) / 256;
  if (nb > 1216) nb = 1216;
  adam_kernel<<<(int)nb, 256, 0, s>>>(n, p, g, a);
  return cudaGetLastError();
}

}  // namespace tnvan
