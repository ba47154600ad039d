// Acceptance and commit: greedy verification (Eq. 4), Relaxed Verification (Eq. 8) and the
// ablation variants (Eq. 7; "top-p" of Section 4.3.2), longest accepted prefix, correction
// or bonus token, and the KV-cache length update.
//
// A row is read once (verdict.cuh), by one CTA or in parts by several: max / arg max (smallest id on
// ties), the tokens ranked ahead of the draft token and, where the rule needs a probability, the
// sum of exp(l - max).  The last CTA of a sequence to finish puts the parts together, walks the rows'
// verdicts in order and writes the outputs.  Reductions have a fixed shape, so results are identical
// from run to run.
#include <algorithm>
#include <mutex>

#include "state.cuh"
#include "verdict.cuh"

namespace laser {
namespace {

constexpr int kAcceptThreads = kVerdictThreads;
constexpr int kMaxAcceptSeqs = 1 << 16;  // counters live at the start of the scratch

// Parts of a row: a CTA goes through its part in batches of 8192 values, a memory round trip each, so rows are cut into two or
// four while all CTAs with work can be resident at once (four an SM).  How many rows are active is known on the device alone: the
// host launches up to twice the CTAs that fit, and the kernel takes so many parts that those with work do.  All rows active,
// relaxed rule, device time in one / two / four parts: 32000 logits, 9 rows 8.7 / 7.3 / 6.8 us, 144 rows 12.9 / 10.5 / 9.6, 288 rows 13.8 /
// 12.0 / 15.0; 12000 logits, 9 rows 6.6 / 6.2 / 6.7, 288 rows 9.9 / 9.2 / 14.8.  Where a whole row takes four batches or more, two parts still
// end sooner with a third more CTAs than fit, and not otherwise: 324 / 396 / 432 rows of 28000 logits 16.4 / 16.4 / 16.5 whole, 14.6 /
// 16.2 / 17.1 in two; of 24000 13.8 / 13.8 / 13.9, 14.5 / 16.2 / 17.0; of 50257 logits 400 / 440 rows 26.5 / 26.7, 25.9 / 27.2.
constexpr int kLaunchedCtas = 8 * 148;
constexpr int kResidentCtas = 4 * 148, kFewCtas = 800, kLongRow = 3 * 8192;
int parts_of(int64_t rows, int32_t V) {
  int parts = 4;
  while (parts > 1 && (rows * parts > kLaunchedCtas || V < 4096 * parts)) parts /= 2;
  return parts;
}

// What the CTAs leave in the scratch: the verdict of a row read whole, or the RowResult of each part.
struct WholeRow { int arg, pass; };
size_t results_bytes(int64_t rows, int parts) {
  return size_t(rows) * std::max(sizeof(WholeRow), parts > 1 ? sizeof(RowResult) * parts : size_t(0));
}

__global__ void __launch_bounds__(kAcceptThreads)
accept_rows_kernel(const float* logits, const int32_t* tokens, const int32_t* n_rows, const int32_t* seq_ids,
                   int32_t R, int32_t V, const Rule rule, int32_t* __restrict__ counters, void* results,
                   int32_t* __restrict__ n_accept, int32_t* __restrict__ out_tokens,
                   int32_t* __restrict__ n_out, int32_t* __restrict__ kv_len, unsigned long long* stamp) {
  const int b = blockIdx.x / R, i = blockIdx.x % R, part = blockIdx.y;
  __shared__ int s_rows;
  if (threadIdx.x == 0) s_rows = 0;
  next_may_launch();
  wait_for_earlier();
  if (stamp && blockIdx.x == 0 && part == 0 && threadIdx.x == 0) *stamp = device_ns();
  const int nr = min(n_rows[b], R);
  const int tid = threadIdx.x;
  int parts = gridDim.y;
  if (parts > 1) {
    int mine = 0;
    for (int x = tid; x < int(gridDim.x) / R; x += kAcceptThreads) mine += min(max(n_rows[x], 0), R);
    __syncthreads();
    mine = __reduce_add_sync(0xffffffffu, mine);
    if ((tid & 31) == 0 && mine) atomicAdd(&s_rows, mine);
    __syncthreads();
    const int few = V > kLongRow ? kFewCtas : kResidentCtas;
    while (parts > 1 && s_rows * parts > few) parts /= 2;
    if (part >= parts) return;
  }
  if (nr <= 0) {
    if (i == 0 && part == 0) {
      if (tid == 0) { n_accept[b] = 0; n_out[b] = 0; }
      for (int j = tid; j < R; j += kAcceptThreads) out_tokens[b * R + j] = -1;
    }
    return;
  }
  if (i >= nr) return;

  // row x verifies draft token x + 1, if there is one
  auto row_of = [&](int x) { return logits + (size_t(b) * R + x) * V; };
  auto token_of = [&](int x) { return x + 1 < nr ? tokens[b * R + x + 1] : -1; };
  RowResult mine = cta_scan(row_of(i), V, part, parts, token_of(i), rule);

  // publish, then let the last CTA of this sequence go through the rows in order
  __shared__ int s_last;
  if (tid == 0) {
    if (parts == 1) {
      const int pass = judge(row_of(i), V, token_of(i), rule, mine);
      static_cast<WholeRow*>(results)[size_t(b) * R + i] = WholeRow{mine.arg, pass};
    } else {
      static_cast<RowResult*>(results)[(size_t(b) * R + i) * parts + part] = mine;
    }
    __threadfence();
    s_last = atomicAdd(&counters[b], 1) == nr * parts - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  __shared__ int s_arg[kAcceptThreads], s_pass[kAcceptThreads];
  int a = 0, base = 0;           // (the same in every thread)
  for (bool go = true;; base += kAcceptThreads) {   // a row a thread: rows base .. base + kAcceptThreads - 1
    const int x = base + tid;
    if (x < nr && parts == 1) {
      const volatile WholeRow* v = static_cast<const WholeRow*>(results) + size_t(b) * R + x;
      s_pass[tid] = v->pass;
      s_arg[tid] = v->arg;
    } else if (x < nr) {
      const volatile RowResult* v = static_cast<const RowResult*>(results) + (size_t(b) * R + x) * parts;
      RowResult r{v->mx, v->arg, v->ahead, v->m, v->s, v->lt};
      for (int q = 1; q < parts; ++q) merge_rows(r, RowResult{v[q].mx, v[q].arg, v[q].ahead, v[q].m, v[q].s, 0.f});
      s_pass[tid] = judge(row_of(x), V, token_of(x), rule, r);
      s_arg[tid] = r.arg;
    }
    __syncthreads();
    for (const int end = min(nr - 1, base + kAcceptThreads); go && a < end; a += go) {
      const int pass = s_pass[a - base];
      go = (pass == 2 ? exact_pass(row_of(a), V, token_of(a), s_arg[a - base], rule.p) : pass) != 0;
    }
    if (!go || a < base + kAcceptThreads) break;
    __syncthreads();
  }
  if (tid == 0) {
    n_accept[b] = a;
    n_out[b] = a + 1;
    if (kv_len) kv_len[seq_ids[b]] += a + 1;
    counters[b] = 0;  // ready for the next call
  }
  for (int j = tid; j < R; j += kAcceptThreads)
    out_tokens[b * R + j] = j < a ? tokens[b * R + j + 1] : (j == a ? s_arg[a - base] : -1);
}

// Fixed scratch of the allocation-free entry point: per-sequence counters, then the rows' results (rows in parts are few).  Its
// size is part of that entry point's contract (laser.h).
constexpr int kNoAllocMaxSeqs = 1024;
constexpr int kNoAllocMaxRows = 16384;
constexpr size_t kNoAllocCounterBytes = sizeof(int32_t) * kNoAllocMaxSeqs;
constexpr size_t kNoAllocBytes = kNoAllocCounterBytes + sizeof(WholeRow) * kNoAllocMaxRows;
static_assert(kNoAllocBytes == 132 * 1024 && kLaunchedCtas * sizeof(RowResult) <= sizeof(WholeRow) * kNoAllocMaxRows, "");
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// Device address of g_noalloc_scratch on the current device, resolved once per device.  Host threads
// may make their first calls at the same time: the table is guarded by a mutex.
laser_status noalloc_scratch(void** out) {
  constexpr int kMaxDevices = 64;
  static void* addr[kMaxDevices] = {};
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  int dev = 0;
  LASER_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) { set_error("device index %d out of range", dev); return LASER_ERR_UNSUPPORTED; }
  if (!addr[dev]) {
    void* p = nullptr;
    // the symbol's name is only a host-side handle; the kernel needs the address the runtime maps it to
    LASER_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    addr[dev] = p;
  }
  *out = addr[dev];
  return LASER_OK;
}

}  // namespace
}  // namespace laser

LASER_API laser_status laser_accept_commit_noalloc(laser_kv* kv, const int32_t* seq_ids, const float* logits,
                                                   const int32_t* tokens, const int32_t* n_rows, int32_t B,
                                                   int32_t V, const laser_params* p, int32_t* n_accept,
                                                   int32_t* out_tokens, int32_t* n_out, void* stream) {
  using namespace laser;
  LASER_REQUIRE(p && logits && tokens && n_rows && n_accept && out_tokens && n_out, "null argument");
  LASER_REQUIRE(B >= 0 && V >= 1 && p->K >= 0, "B = %d, V = %d, K = %d", B, V, p->K);
  LASER_REQUIRE(p->mode >= LASER_MODE_STRICT && p->mode <= LASER_MODE_RELAXED_ARGMAX, "mode = %d", p->mode);
  LASER_REQUIRE(p->mode == LASER_MODE_STRICT || p->mode == LASER_MODE_TOPP || p->topk >= 1, "topk = %d", p->topk);
  LASER_REQUIRE(kv == nullptr || seq_ids != nullptr, "seq_ids is required when committing");
  const int64_t rows = int64_t(B) * (int64_t(p->K) + 1);
  if (B > kNoAllocMaxSeqs || rows > kNoAllocMaxRows) {
    set_error("laser_accept_commit_noalloc handles at most %d sequences and %d rows (B * (K+1)); got B = %d, rows = %lld",
              kNoAllocMaxSeqs, kNoAllocMaxRows, B, (long long)rows);
    return LASER_ERR_CAPACITY;
  }
  if (B == 0) return LASER_OK;
  void* scratch = nullptr;
  LASER_TRY(noalloc_scratch(&scratch));
  int32_t* counters = static_cast<int32_t*>(scratch);
  void* results = static_cast<char*>(scratch) + kNoAllocCounterBytes;
  // the array keeps whatever the previous call left: the arrival counters must start at zero
  LASER_CUDA(cudaMemsetAsync(counters, 0, sizeof(int32_t) * size_t(B), as_stream(stream)));
  const int R = p->K + 1, parts = parts_of(rows, V);
  LASER_CUDA(launch_overlapped(accept_rows_kernel, dim3(unsigned(B * R), unsigned(parts)), kAcceptThreads, 0, as_stream(stream),
      logits, tokens, n_rows, seq_ids, R, V, Rule{p->mode, p->topk, double(p->p)}, counters, results,
      n_accept, out_tokens, n_out, kv ? kv->seq_len : nullptr, static_cast<unsigned long long*>(nullptr)));
  count_launch();
  LASER_CUDA(cudaGetLastError());
  return LASER_OK;
}

namespace laser {
laser_status accept_commit(laser_kv* kv, const int32_t* seq_ids, const float* logits, const int32_t* tokens, const int32_t* n_rows,
                           int32_t B, int32_t V, const laser_params* p, int32_t* n_accept, int32_t* out_tokens, int32_t* n_out,
                           unsigned long long* stamp, cudaStream_t stream) {
  LASER_REQUIRE(p && logits && tokens && n_rows && n_accept && out_tokens && n_out, "null argument");
  LASER_REQUIRE(B >= 0 && B <= kMaxAcceptSeqs, "B = %d outside [0, %d]", B, kMaxAcceptSeqs);
  LASER_REQUIRE(V >= 1, "V = %d", V);
  LASER_REQUIRE(p->K >= 0 && p->K <= 1023, "K = %d outside [0, 1023]", p->K);
  LASER_REQUIRE(p->mode >= LASER_MODE_STRICT && p->mode <= LASER_MODE_RELAXED_ARGMAX, "mode = %d", p->mode);
  LASER_REQUIRE(p->mode == LASER_MODE_STRICT || p->mode == LASER_MODE_TOPP || p->topk >= 1,
                "topk = %d", p->topk);
  LASER_REQUIRE(kv == nullptr || seq_ids != nullptr, "seq_ids is required when committing");
  if (B == 0) return LASER_OK;
  const int R = p->K + 1, parts = parts_of(int64_t(B) * R, V);
  void* scratch = nullptr;
  const size_t counters_bytes = sizeof(int32_t) * kMaxAcceptSeqs;
  LASER_TRY(scratch_get(SCRATCH_ACCEPT, counters_bytes + results_bytes(int64_t(B) * R, parts), &scratch));
  int32_t* counters = static_cast<int32_t*>(scratch);
  void* results = static_cast<char*>(scratch) + counters_bytes;
  LASER_CUDA(launch_overlapped(accept_rows_kernel, dim3(unsigned(B * R), unsigned(parts)), kAcceptThreads, 0, stream,
      logits, tokens, n_rows, seq_ids, R, V, Rule{p->mode, p->topk, double(p->p)}, counters, results,
      n_accept, out_tokens, n_out, kv ? kv->seq_len : nullptr, stamp));
  count_launch();
  LASER_CUDA(cudaGetLastError());
  return LASER_OK;
}
}  // namespace laser

LASER_API laser_status laser_accept_commit(laser_kv* kv, const int32_t* seq_ids,
                                           const float* logits, const int32_t* tokens,
                                           const int32_t* n_rows, int32_t B, int32_t V,
                                           const laser_params* p, int32_t* n_accept,
                                           int32_t* out_tokens, int32_t* n_out, void* stream) {
  return laser::accept_commit(kv, seq_ids, logits, tokens, n_rows, B, V, p, n_accept, out_tokens, n_out, nullptr, laser::as_stream(stream));
}
