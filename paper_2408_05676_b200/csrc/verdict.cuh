// Row pass shared by the acceptance kernels (Eq. 4, Eq. 7, Eq. 8 and the variants of Section 4.3.2): max and arg max of a row
// of logits, and the verdict on one token given its row - its rank (tokens ahead of it; equal logits rank the smaller id
// first) and, where the rule needs it, whether its probability exceeds p, the denominator in fp64 from fp32 differences.
// One CTA of kVerdictThreads threads works on one row or a part of it; reductions have a fixed shape, so results are identical from
// run to run.
//
// The row is read once, 16 bytes a load and eight loads in flight per thread.  The probability is first estimated in fp32 with a
// running maximum; the fp64 sum - an exponential per token, which used to be most of the kernel - is taken only where the
// estimate lies within its error bound of p, so that the verdict is always the fp64 one.  64 sequences x 1 .. 9 rows of 32000
// logits, relaxed rule: 57.5 -> 20.1 us; 18.4 with launches overlapped, 17.6 with the rows in two parts each, 16.7 with sums that take
// the same steps whether there is a maximum yet or not.
#pragma once
#include "common.cuh"

namespace laser {

constexpr int kVerdictThreads = 256;
constexpr int kRowLoads = 8;       // float4 loads in flight per thread

__device__ __forceinline__ void better(float& v, int& i, float ov, int oi) {
  if (ov > v || (ov == v && oi < i)) { v = ov; i = oi; }
}

constexpr int kNoId = 0x7fffffff;   // no arg max (a row of NaN alone)

struct RowResult { float mx; int arg; int ahead; float m, s, lt; };   // s = sum of exp(x - m) over what was seen; lt = the token's

// exp(d) for d <= 0.  ex2 is good to 2 units in the last place and the product's rounding shifts the exponent by |d| 2^-24:
// within 1e-5 of exp(d) wherever that is not below 1e-38.
__device__ __forceinline__ float exp_below(float d) { return exp2f(d * 1.4426950408889634f); }

template <bool RANK, bool PROB>
__device__ __forceinline__ RowResult scan_row(const float* __restrict__ row, int V, int part, int parts, int t, float lt, int tid) {
  RowResult r{-INFINITY, kNoId, 0, -INFINITY, 0.f, lt};
  const int lead = min(V, int((16 - (reinterpret_cast<uintptr_t>(row) & 15)) & 15) >> 2);   // values before the first 16-byte boundary
  const int n4 = (V - lead) >> 2;
  // cnt values and their ids; equal logits rank ahead of the token where their id is below `before` (padding, -inf, must not be)
  auto batch = [&](const float* x, int cnt, auto index_of, int before) {
    float bm = -INFINITY;
#pragma unroll
    for (int i = 0; i < cnt; ++i) bm = fmaxf(bm, x[i]);
    if (bm > r.mx || r.arg == kNoId) {   // ids ascend from batch to batch and inside one: the first of equals stays
      r.mx = bm;
#pragma unroll
      for (int i = cnt - 1; i >= 0; --i) if (x[i] == bm) r.arg = index_of(i);
    }
    if (RANK) {
      bool eq = false;
#pragma unroll
      for (int i = 0; i < cnt; ++i) { r.ahead += x[i] > lt; eq |= x[i] == lt; }
      if (eq)
#pragma unroll
        for (int i = 0; i < cnt; ++i) r.ahead += x[i] == lt && index_of(i) < before;
    }
    if (PROB) {
      if (bm > r.m) { r.s *= r.m > -INFINITY ? exp_below(r.m - bm) : 0.f; r.m = bm; }   // (a NaN stays)
      const float ref = r.m > -INFINITY ? r.m : 0.f;   // (nothing above -inf so far: the terms are 0, or NaN)
      float add = 0.f;
#pragma unroll
      for (int i = 0; i < cnt; ++i) add += exp_below(x[i] - ref);
      r.s += add;
    }
  };
  const int per = (n4 + parts - 1) / parts, end = min(n4, (part + 1) * per);   // (float4s of this part: part * per .. end - 1)
  if (part == 0 && tid < lead) batch(row + tid, 1, [&](int) { return tid; }, t);
  const float4* r4 = reinterpret_cast<const float4*>(row + lead);
  for (int base = part * per; base < end; base += kVerdictThreads * kRowLoads) {
    float x[4 * kRowLoads];
#pragma unroll
    for (int u = 0; u < kRowLoads; ++u) {
      const int i = base + u * kVerdictThreads + tid;
      const float4 v = i < end ? r4[i] : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      x[4 * u] = v.x; x[4 * u + 1] = v.y; x[4 * u + 2] = v.z; x[4 * u + 3] = v.w;
    }
    batch(x, 4 * kRowLoads, [&](int i) { return lead + 4 * (base + (i >> 2) * kVerdictThreads + tid) + (i & 3); }, min(t, lead + 4 * end));
  }
  if (r.arg >= lead + 4 * end) r.arg = kNoId;   // (padding, where nothing was above -inf)
  const int tail = lead + 4 * n4 + tid;
  if (part == parts - 1 && tail < V) batch(row + tail, 1, [&](int) { return tail; }, t);
  return r;
}

__device__ __forceinline__ void merge_rows(RowResult& r, const RowResult& o) {
  better(r.mx, r.arg, o.mx, o.arg);
  r.ahead += o.ahead;
  const float m = fmaxf(r.m, o.m), ref = m > -INFINITY ? m : 0.f;   // (a sum without a maximum is 0 or NaN)
  r.s = r.s * exp_below(r.m - ref) + o.s * exp_below(o.m - ref);
  r.m = m;
}

struct Rule {
  int mode, topk;
  double p;
  __device__ bool needs_p() const { return mode == LASER_MODE_RELAXED || mode == LASER_MODE_TOPP || mode == LASER_MODE_RELAXED_ARGMAX; }
  __device__ bool needs_rank() const { return mode == LASER_MODE_RELAXED || mode == LASER_MODE_TOPK || mode == LASER_MODE_RELAXED_ARGMAX; }
};

// What a CTA finds in its part of a row, in thread 0.  t: the token whose verdict the row gives (t < 0: none).
static __device__ RowResult cta_scan(const float* row, int V, int part, int parts, int t, const Rule& rule) {
  constexpr int kWarps = kVerdictThreads / 32;
  __shared__ RowResult s_part[kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool judged = t >= 0 && t < V;
  const bool need_p = judged && rule.needs_p(), need_rank = judged && rule.needs_rank();
  const float lt = judged ? row[t] : 0.f;
  RowResult r = need_p ? (need_rank ? scan_row<true, true>(row, V, part, parts, t, lt, tid) : scan_row<false, true>(row, V, part, parts, t, lt, tid))
                       : (need_rank ? scan_row<true, false>(row, V, part, parts, t, lt, tid) : scan_row<false, false>(row, V, part, parts, t, lt, tid));
  for (int o = 16; o; o >>= 1) {
    RowResult other;
    other.mx = __shfl_xor_sync(0xffffffffu, r.mx, o);
    other.arg = __shfl_xor_sync(0xffffffffu, r.arg, o);
    other.ahead = __shfl_xor_sync(0xffffffffu, r.ahead, o);
    other.m = __shfl_xor_sync(0xffffffffu, r.m, o);
    other.s = __shfl_xor_sync(0xffffffffu, r.s, o);
    merge_rows(r, other);
  }
  __syncthreads();   // the shared slots may still be read from an earlier call
  if (lane == 0) s_part[warp] = r;
  __syncthreads();
  if (tid == 0)
    for (int w = 1; w < kWarps; ++w) merge_rows(r, s_part[w]);
  return r;
}

// One thread, from a whole row's result: the arg max (smallest id on ties), and whether t passes: 0, 1, or 2 where only the rule's
// own arithmetic (exact_pass) can tell.
static __device__ int judge(const float* row, int V, int t, const Rule& rule, const RowResult& r) {
  if (t < 0 || t >= V) return 0;
  const bool top = t == r.arg, in_topk = r.ahead < rule.topk;
  // The estimate's relative error: each term 1e-5, a term's at most 6 rescalings per thread (V / 8192 batches; rows beyond
  // 49152 tokens add one per 8192) and 8 + 7 merges (lanes and warps, parts) 1e-5 each, sums of 128 + 20 terms 1e-5; the numerator
  // 1e-5.  Twice that.
  const double margin = 5.2e-4 + 2e-9 * V;
  const double q = double(exp_below(r.lt - r.mx)) / double(r.s);
  const bool estimated = rule.p <= 0.0 || rule.p >= 1e-30;   // (a probability near a smaller p has lost digits in fp32)
  const bool matters = rule.needs_p() && (rule.mode == LASER_MODE_RELAXED ? in_topk : rule.mode == LASER_MODE_TOPP ? !top : !top && in_topk);
  const bool sure_above = q * (1.0 - margin) > rule.p, sure_below = q * (1.0 + margin) < rule.p;
  if (matters && !(estimated && (sure_above || sure_below))) return 2;      // (a NaN is neither)
  if (rule.mode == LASER_MODE_STRICT) return top;
  if (rule.mode == LASER_MODE_RELAXED) return in_topk && sure_above;
  if (rule.mode == LASER_MODE_TOPK) return in_topk;
  if (rule.mode == LASER_MODE_RELAXED_ARGMAX) return top || (in_topk && sure_above);
  return top || sure_above;
}

// The rule's own arithmetic, by the whole CTA: everything else about the row (whose arg max is given) is settled, the
// probability decides.  Every thread gets the answer.
static __device__ int exact_pass(const float* row, int V, int t, int arg, double p) {
  constexpr int kWarps = kVerdictThreads / 32;
  __shared__ double s_sum[kWarps];
  __shared__ int s_pass;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float mx = arg < V ? row[arg] : -INFINITY;   // (no arg max: nothing but NaN)
  double sum = 0.0;
  for (int j = tid; j < V; j += kVerdictThreads) sum += exp(double(row[j] - mx));
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  __syncthreads();   // (the slots of an earlier call)
  if (lane == 0) s_sum[warp] = sum;
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < kWarps; ++w) sum += s_sum[w];
    s_pass = exp(double(row[t] - mx)) / sum > p;
  }
  __syncthreads();
  return s_pass;
}

// Max and arg max (smallest id on ties) of a row, and whether token t passes on it (t < 0: none), in every thread.
static __device__ void cta_row(const float* row, int V, int t, const Rule& rule, int* arg_out, int* pass_out) {
  __shared__ int s_arg, s_verdict;
  RowResult r = cta_scan(row, V, 0, 1, t, rule);
  if (threadIdx.x == 0) {
    s_verdict = judge(row, V, t, rule, r);
    s_arg = r.arg;
  }
  __syncthreads();
  *arg_out = s_arg;
  const int verdict = s_verdict;
  *pass_out = verdict == 2 ? exact_pass(row, V, t, s_arg, rule.p) : verdict;
}

}  // namespace laser
