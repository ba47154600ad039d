// Generation loop: Draft-Then-Verify decoding (Section 2.1, Section 3) and, with no pool,
// plain greedy autoregressive decoding (Eq. 1).  All per-step state stays on the device; after a
// step the device reports to pinned host memory how many sequences are still active and how far
// the furthest of them has to go, and the host queues the next steps from that.
#include <string.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "model.cuh"

namespace laser {
namespace {

// What a step tells the host, in one 64-bit store: the tokens that the furthest sequence has to go (0: all are finished), the
// error word, and a tag by which the host knows the step.
__host__ __device__ inline unsigned long long report_of(int remaining, int status, unsigned tag) {
  return (unsigned long long)(unsigned(remaining)) << 32 | (unsigned long long)(unsigned(status) & 0xffu) << 24 | (tag & 0xffffffu);
}

enum { COUNT_STEPS = 0, COUNT_DRAFTED, COUNT_ACCEPTED, COUNT_EMITTED, NS_DRAFT, NS_VERIFY, NS_ACCEPT, COUNTERS };
enum { STAMP_END = 0, STAMP_DRAFTED, STAMP_START, STAMP_VERIFIED, STAMPS };   // device clock: the step before ended, ...

struct GenState {
  int32_t* seq_tok;      // [B, max_total] prompt followed by generated tokens
  int32_t* seq_len;      // [B] tokens in seq_tok
  int32_t* done;         // [B]
  unsigned long long* counters;  // [COUNTERS]
  unsigned long long* stamps;    // [STAMPS]
  int32_t* out_len;      // [B] generated so far
  int32_t* out;          // [B, max_new]
  int32_t *tails, *tail_len, *last;   // of the next step: last n_max tokens (right-aligned), their number, the pending token
  int32_t* kv_len;       // the cache's committed lengths
  const int32_t* status; // the model's error word
  int B, Rs, max_total, max_new, n_max, eos;
};

// Ends a step and prepares the next: truncates the emitted tokens to the room left, stops at EOS, appends, advances the
// cache, and leaves the tail and the pending token of every active sequence (none once an error is pending).  `first`: only
// the preparation, and the cache's lengths after the prompts.  One block, a warp per sequence in turn: the work is a few
// dependent loads, and one launch of it between two steps is what it costs.  `fused`: the verdict came with the forward.
constexpr int kStepThreads = 1024;
__global__ void __launch_bounds__(kStepThreads)
step_kernel(const GenState g, int first, int fused, const int32_t* n_rows, const int32_t* n_accept, const int32_t* out_tokens,
            const int32_t* n_out, volatile unsigned long long* report, unsigned tag) {
  __shared__ int s_remaining;
  __shared__ unsigned long long s_count[4];
  next_may_launch();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x < 4) s_count[threadIdx.x] = 0;
  if (threadIdx.x == 0) s_remaining = 0;
  __syncthreads();
  wait_for_earlier();
  const unsigned long long entered = device_ns();
  const int bad = *g.status;
  for (int b = warp; b < g.B; b += kStepThreads / 32) {
    bool done = g.done[b] != 0;
    int len = g.seq_len[b], made = g.out_len[b];
    int32_t* text = g.seq_tok + size_t(b) * g.max_total;
    const int rows = first ? 0 : n_rows[b];
    if (first && lane == 0) g.kv_len[b] = len - 1;
    if (!done && rows > 0) {
      int n = min(n_out[b], g.max_new - made);
      const int32_t* emitted = out_tokens + b * g.Rs;
      for (int j0 = 0; g.eos >= 0 && j0 < n; j0 += 32) {
        const unsigned hit = __ballot_sync(0xffffffffu, j0 + lane < n && emitted[j0 + lane] == g.eos);
        if (hit) { n = j0 + __ffs(hit); done = true; }
      }
      for (int j = lane; j < n; j += 32) {
        const int32_t t = emitted[j];
        g.out[size_t(b) * g.max_new + made + j] = t;
        text[len + j] = t;
      }
      len += n;
      made += n;
      done = done || made >= g.max_new;
      if (lane == 0) {
        g.out_len[b] = made; g.seq_len[b] = len; g.kv_len[b] += n; g.done[b] = done;
        atomicAdd(&s_count[0], 1ULL);
        atomicAdd(&s_count[1], (unsigned long long)(rows - 1));
        atomicAdd(&s_count[2], (unsigned long long)n_accept[b]);
        atomicAdd(&s_count[3], (unsigned long long)n);
      }
      __syncwarp();
    }
    if (!done && lane == 0) atomicMax(&s_remaining, g.max_new - made);
    const bool stop = done || bad;
    const int tl = stop ? 0 : min(g.n_max, len);
    if (lane < g.n_max) g.tails[b * g.n_max + lane] = lane >= g.n_max - tl ? text[len - g.n_max + lane] : -1;
    if (lane == 0) { g.tail_len[b] = tl; g.last[b] = stop ? -1 : text[len - 1]; }
  }
  __syncthreads();
  if (threadIdx.x < 4 && s_count[threadIdx.x]) g.counters[threadIdx.x] += s_count[threadIdx.x];
  if (threadIdx.x == 0) {
    const unsigned long long ended = device_ns();
    if (!first) {
      *report = report_of(s_remaining, bad, tag);
      const unsigned long long verified = fused ? entered : g.stamps[STAMP_VERIFIED];
      g.counters[NS_DRAFT] += g.stamps[STAMP_DRAFTED] - g.stamps[STAMP_END];
      g.counters[NS_VERIFY] += verified - max(g.stamps[STAMP_START], g.stamps[STAMP_DRAFTED]);
      g.counters[NS_ACCEPT] += ended - verified;
    }
    g.stamps[STAMP_END] = ended;
  }
}

__global__ void stamp_kernel(unsigned long long* stamp) {
  wait_for_earlier();
  *stamp = device_ns();
}

__global__ void no_draft_kernel(int B, int K, int32_t* __restrict__ draft, int32_t* __restrict__ draft_len) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < B * K) draft[i] = -1;
  if (i < B) draft_len[i] = 0;
}

// Work buffers of one laser_generate call, carved out of one allocation that the model keeps and only
// ever grows: requests are collected first, then placed, 256-byte aligned.
struct DevBuf {
  struct Req { void** p; size_t bytes; };
  std::vector<Req> reqs;
  template <typename T>
  void get(T** p, size_t count) {
    reqs.push_back(Req{reinterpret_cast<void**>(p), std::max<size_t>(count, 1) * sizeof(T)});
  }
  laser_status commit(laser_model* m, cudaStream_t stream) {
    size_t total = 0;
    for (const Req& r : reqs) total += (r.bytes + 255) & ~size_t(255);
    if (total > m->gen_bytes) {
      LASER_CUDA(cudaStreamSynchronize(stream));
      if (m->gen_buf) {
        LASER_CUDA(cudaFree(m->gen_buf));
        m->owned.erase(std::remove(m->owned.begin(), m->owned.end(), m->gen_buf), m->owned.end());
      }
      m->gen_buf = nullptr; m->gen_bytes = 0;
      LASER_CUDA(device_malloc(&m->gen_buf, total));
      m->owned.push_back(m->gen_buf);
      m->gen_bytes = total;
    }
    size_t off = 0;
    for (const Req& r : reqs) { *r.p = static_cast<char*>(m->gen_buf) + off; off += (r.bytes + 255) & ~size_t(255); }
    return LASER_OK;
  }
};

// A prompt's tokens start .. start + rows - 1, and the chunks of a pass in the order in which attention takes them: kPrefillShare
// consecutive chunks of a prompt at a time, those that see most keys first (its CTAs differ by the keys that they walk, and one that
// starts last and walks longest is what the launch would end with).  What a prompt has beyond a multiple of kPrefillShare is the
// beginning of its part of the pass, which sees least, and goes behind all others.
struct Chunk { int prompt, start, rows; };
void order_pass(Chunk* pass, int n) {
  struct Run { int first, n, keys; };
  std::vector<Run> runs;
  for (int c = 0; c < n;) {
    int e = c;
    while (e < n && pass[e].prompt == pass[c].prompt) ++e;
    for (int x = c, take; x < e; x += take) {
      take = (e - x) % kPrefillShare ? (e - x) % kPrefillShare : kPrefillShare;
      runs.push_back(Run{x, take, pass[x + take - 1].start + pass[x + take - 1].rows});
    }
    c = e;
  }
  std::stable_sort(runs.begin(), runs.end(), [](const Run& a, const Run& b) {
    return (a.n == kPrefillShare) != (b.n == kPrefillShare) ? a.n == kPrefillShare : a.keys > b.keys;
  });
  std::vector<Chunk> out;
  out.reserve(size_t(n));
  for (const Run& r : runs) out.insert(out.end(), pass + r.first, pass + r.first + r.n);
  std::copy(out.begin(), out.end(), pass);
}

constexpr int kInFlight = 2;   // steps queued beyond the last whose report has been read
constexpr int kSlots = 4;      // reports

}  // namespace

// The host's side of the loop, kept with the model: pinned memory for the calls' inputs, results and the steps' reports.
struct GenHost {
  char* pinned = nullptr;
  size_t bytes = 0;
  volatile unsigned long long* report = nullptr;   // [kSlots]
  unsigned tag = 1;                                // of the next step, over all calls: what a failed call left behind is told apart
  cudaEvent_t uploaded = nullptr, begin = nullptr, prefilled = nullptr;

  ~GenHost() {
    if (pinned) cudaFreeHost(pinned);
    if (report) cudaFreeHost(const_cast<unsigned long long*>(report));
    for (cudaEvent_t e : {uploaded, begin, prefilled}) if (e) cudaEventDestroy(e);
  }
  laser_status open() {
    LASER_CUDA(cudaEventCreateWithFlags(&uploaded, cudaEventDisableTiming));
    LASER_CUDA(cudaEventCreate(&begin));
    LASER_CUDA(cudaEventCreate(&prefilled));
    void* r = nullptr;
    LASER_CUDA(cudaHostAlloc(&r, sizeof(unsigned long long) * kSlots, cudaHostAllocDefault));
    memset(r, 0, sizeof(unsigned long long) * kSlots);
    report = static_cast<volatile unsigned long long*>(r);
    return LASER_OK;
  }
  // The report of the step tagged `t`: read where the device writes it (an event behind the step would keep the next kernel
  // from overlapping).  Ends when the stream has nothing left to run, or failed.
  laser_status wait_report(unsigned t, cudaStream_t stream, unsigned long long* out) {
    for (unsigned spin = 1;; ++spin) {
      const unsigned long long r = report[t % kSlots];
      if ((r & 0xffffffu) == (t & 0xffffffu)) { *out = r; std::atomic_thread_fence(std::memory_order_acquire); return LASER_OK; }
      if (spin % 4096) continue;
      const cudaError_t e = cudaStreamQuery(stream);
      if (e == cudaErrorNotReady) continue;
      LASER_CUDA(e);
      if ((report[t % kSlots] & 0xffffffu) != (t & 0xffffffu)) { set_error("a generation step ended without its report"); return LASER_ERR_CUDA; }
    }
  }
  // pinned memory of at least `n` bytes, once the copies out of it that an earlier call queued are over
  laser_status pinned_get(size_t n, char** out) {
    LASER_CUDA(cudaEventSynchronize(uploaded));
    if (n > bytes) {
      if (pinned) LASER_CUDA(cudaFreeHost(pinned));
      pinned = nullptr; bytes = 0;
      LASER_CUDA(cudaHostAlloc(reinterpret_cast<void**>(&pinned), n, cudaHostAllocDefault));
      bytes = n;
    }
    *out = pinned;
    return LASER_OK;
  }
};

void gen_host_free(laser_model* m) {
  delete m->gen_host;
  m->gen_host = nullptr;
}

}  // namespace laser

using namespace laser;

LASER_API laser_status laser_generate(laser_model* m, laser_kv* kv, const laser_pool* pool, const int32_t* prompts,
                                      const int64_t* prompt_offsets, const int32_t* group_id, int32_t B,
                                      const laser_params* p, int32_t* out, int32_t* out_len, laser_stats* stats,
                                      void* stream_) {
  LASER_REQUIRE(m && kv && prompts && prompt_offsets && p && out && out_len, "null argument");
  LASER_REQUIRE(pool == nullptr || group_id != nullptr, "group_id is required with a pool");
  LASER_REQUIRE(B >= 1 && B <= m->cfg.max_batch && B <= kv->max_seqs, "B = %d outside [1, min(max_batch, max_seqs)]", B);
  LASER_REQUIRE(p->K == m->cfg.max_draft, "params K = %d differs from the model's max_draft = %d", p->K, m->cfg.max_draft);
  LASER_REQUIRE(p->max_new >= 1, "max_new = %d", p->max_new);
  LASER_REQUIRE(pool == nullptr || (p->K >= 1 && p->n_max >= 1 && p->n_max <= 8), "drafting needs K >= 1 and n_max in [1, 8]");
  LASER_REQUIRE(!p->temp_branches || pool != nullptr, "temporary branches are drafted beside a pool");
  LASER_REQUIRE(!p->tree || pool != nullptr, "tree drafting needs a pool");
  cudaStream_t stream = as_stream(stream_);
  const int K = p->K, Rs = K + 1, n_max = pool ? p->n_max : 1;
  int max_prompt = 0, n_chunks = 0;
  for (int b = 0; b < B; ++b) {
    const int64_t len = prompt_offsets[b + 1] - prompt_offsets[b];
    LASER_REQUIRE(len >= 1, "prompt %d is empty", b);
    LASER_REQUIRE(len - 1 + p->max_new + K <= kv->capacity_tokens(),
                  "prompt %d (%lld tokens) + max_new + K does not fit the %lld tokens of its KV pages", b,
                  (long long)len, (long long)kv->capacity_tokens());
    max_prompt = std::max<int>(max_prompt, int(len));
    n_chunks += int((len - 1 + kPrefillChunk - 1) / kPrefillChunk);
  }
  const long long launches0 = g_launches;
  const int max_total = max_prompt + p->max_new + Rs;
  if (!m->gen_host) {
    m->gen_host = new GenHost();
    const laser_status st = m->gen_host->open();
    if (st != LASER_OK) { gen_host_free(m); return st; }
  }
  GenHost& host = *m->gen_host;

  // What the host sets goes up in one copy, and the results come back in one: counters, generated lengths | tokens, text
  // lengths, done flags, slots, groups, texts, prefill chunks.  Of those chunks (every prompt token but the last):
  // [chunks][kPrefillChunk] tokens, then per chunk its slot, its first position and its rows.
  size_t words = 0;
  auto part = [&](size_t n) { const size_t at = words; words += (n + 3) & ~size_t(3); return at; };
  const size_t at_counters = part(2 * COUNTERS), at_stamps = part(2 * STAMPS), at_out_len = part(B), at_out = part(size_t(B) * p->max_new), n_result = words;
  const size_t at_len = part(B), at_done = part(B), at_ids = part(B), at_gid = part(B), at_text = part(size_t(B) * max_total),
               at_pre = part(size_t(n_chunks) * (kPrefillChunk + 3));
  char* pinned = nullptr;
  LASER_TRY(host.pinned_get(words * 4, &pinned));
  int32_t* h = reinterpret_cast<int32_t*>(pinned);
  memset(h, 0, at_out * 4);
  memset(h + at_out, 0xff, (n_result - at_out) * 4);
  memset(h + at_done, 0, size_t(B) * 4);
  int32_t *h_pre = h + at_pre, *h_slot = h_pre + size_t(n_chunks) * kPrefillChunk, *h_start = h_slot + n_chunks, *h_rows = h_start + n_chunks;
  std::vector<Chunk> chunks;
  chunks.reserve(size_t(n_chunks));
  for (int b = 0; b < B; ++b) {
    const int len = int(prompt_offsets[b + 1] - prompt_offsets[b]);
    h[at_len + b] = len;
    h[at_ids + b] = b;
    h[at_gid + b] = pool ? group_id[b] : -1;
    int32_t* text = h + at_text + size_t(b) * max_total;
    memcpy(text, prompts + prompt_offsets[b], size_t(len) * 4);
    memset(text + len, 0, size_t(max_total - len) * 4);
    for (int p0 = 0; p0 < len - 1; p0 += kPrefillChunk) chunks.push_back(Chunk{b, p0, std::min(kPrefillChunk, len - 1 - p0)});
  }
  const std::vector<int> passes = prefill_passes(m, n_chunks);
  for (int c0 = 0, i = 0; c0 < n_chunks; c0 += passes[size_t(i++)]) order_pass(chunks.data() + c0, passes[size_t(i)]);
  for (int c = 0; c < n_chunks; ++c) {
    const Chunk& x = chunks[size_t(c)];
    int32_t* row = h_pre + size_t(c) * kPrefillChunk;
    memcpy(row, prompts + prompt_offsets[x.prompt] + x.start, size_t(x.rows) * 4);
    std::fill(row + x.rows, row + kPrefillChunk, -1);
    h_slot[c] = x.prompt; h_start[c] = x.start; h_rows[c] = x.rows;
  }

  DevBuf buf;
  GenState g{};
  int32_t *init, *tokens, *n_rows, *draft, *draft_len, *match_n, *n_accept, *out_tokens, *n_out, *draft_par, *parents, *path_rows;
  float* logits;
  buf.get(&init, words);
  buf.get(&tokens, size_t(B) * Rs);
  buf.get(&n_rows, size_t(B));
  buf.get(&g.tails, size_t(B) * n_max);
  buf.get(&g.tail_len, size_t(B));
  buf.get(&g.last, size_t(B));
  buf.get(&draft, size_t(B) * std::max(K, 1));
  buf.get(&draft_len, size_t(B));
  buf.get(&match_n, size_t(B));
  buf.get(&draft_par, size_t(B) * std::max(K, 1));
  buf.get(&parents, size_t(B) * Rs);
  buf.get(&path_rows, size_t(B) * Rs);
  buf.get(&n_accept, size_t(B));
  buf.get(&out_tokens, size_t(B) * Rs);
  buf.get(&n_out, size_t(B));
  const bool tree = pool && p->tree, fused = p->fused_accept && !tree;   // fused: chain steps without stored logits
  buf.get(&logits, fused ? size_t(4) : size_t(B) * Rs * m->cfg.vocab);
  LASER_TRY(buf.commit(m, stream));
  g.counters = reinterpret_cast<unsigned long long*>(init + at_counters);
  g.stamps = reinterpret_cast<unsigned long long*>(init + at_stamps);
  g.out_len = init + at_out_len; g.out = init + at_out;
  g.seq_len = init + at_len; g.done = init + at_done; g.seq_tok = init + at_text;
  const int32_t *seq_ids = init + at_ids, *gid = init + at_gid;
  g.kv_len = kv->seq_len; g.status = m->status;
  g.B = B; g.Rs = Rs; g.max_total = max_total; g.max_new = p->max_new; g.n_max = n_max; g.eos = p->eos_id;

  LASER_CUDA(cudaMemcpyAsync(init, h, words * 4, cudaMemcpyHostToDevice, stream));
  LASER_CUDA(cudaEventRecord(host.uploaded, stream));
  LASER_CUDA(cudaEventRecord(host.begin, stream));
  // A pass takes chunks of whatever prompts; what a prompt has in several passes comes in order.
  const int32_t *pre = init + at_pre, *slot = pre + size_t(n_chunks) * kPrefillChunk, *start = slot + n_chunks, *rows = start + n_chunks;
  int c0 = 0, n_pass = 0;
  for (const int pass : passes) {
    LASER_TRY(prefill_chunks(m, kv, slot + c0, start + c0, pre + size_t(c0) * kPrefillChunk, rows + c0, pass, stream));
    c0 += pass;
    if ((n_pass++ & 15) == 15) LASER_TRY(laser_check(m, stream));   // do not keep launching after a device-side error
  }
  LASER_CUDA(cudaEventRecord(host.prefilled, stream));
  LASER_CUDA(launch_overlapped(step_kernel, dim3(1), kStepThreads, 0, stream, g, 1, 0, n_rows, n_accept, out_tokens, n_out, host.report, 0u));
  count_launch();
  if (!pool) {   // no drafts, in no step
    no_draft_kernel<<<ceil_div(B * std::max(K, 1), 128), 128, 0, stream>>>(B, K, draft, draft_len);
    count_launch();
  }

  laser_params acc = *p;
  // the drafts of the next step and the rows they make
  auto queue_draft = [&]() -> laser_status {
    if (pool) {
      // temporary branch: the sequence's prompt and generated tokens (seq_tok) are searched as well
      if (p->tree)
        LASER_TRY(laser_draft_tree(pool, g.tails, g.tail_len, gid, p->temp_branches ? g.seq_tok : nullptr,
                                   p->temp_branches ? g.seq_len : nullptr, p->temp_branches ? max_total : 0, B, p, draft,
                                   draft_par, draft_len, match_n, stream));
      else if (p->temp_branches)
        LASER_TRY(laser_draft_temp(pool, g.tails, g.tail_len, gid, g.seq_tok, g.seq_len, max_total, B, p, draft, draft_len,
                                   match_n, stream));
      else
        LASER_TRY(laser_draft(pool, g.tails, g.tail_len, gid, B, p, draft, draft_len, match_n, stream));
    }
    if (tree) return make_rows_tree(g.last, draft, draft_par, draft_len, B, K, tokens, parents, n_rows, g.stamps + STAMP_DRAFTED, stream);
    return make_rows(g.last, draft, draft_len, B, K, tokens, n_rows, g.stamps + STAMP_DRAFTED, stream);
  };
  // the rest of a step: verify, accept, commit; `idle` = the device may have run out of work before it
  auto queue_step = [&](unsigned tag, bool idle) -> laser_status {
    if (idle) {
      LASER_CUDA(launch_overlapped(stamp_kernel, dim3(1), 1, 0, stream, g.stamps + STAMP_START));
      count_launch();
    }
    if (tree) LASER_TRY(laser_verify_step_tree(m, kv, seq_ids, tokens, parents, n_rows, B, logits, stream));
    else if (fused) LASER_TRY(laser_verify_accept(m, kv, seq_ids, tokens, n_rows, B, &acc, 0, nullptr, n_accept, out_tokens, n_out, stream));
    else LASER_TRY(laser_verify_step(m, kv, seq_ids, tokens, n_rows, B, logits, stream));
    if (tree) {
      // verdict, then the accepted path's K/V to consecutive slots (the lengths advance in step_kernel)
      LASER_TRY(accept_tree(nullptr, nullptr, logits, tokens, parents, n_rows, B, m->cfg.vocab, &acc, n_accept, out_tokens, n_out,
                            path_rows, g.stamps + STAMP_VERIFIED, stream));
      LASER_TRY(laser_kv_compact_path(kv, seq_ids, path_rows, n_accept, B, Rs, stream));
    } else if (!fused) {   // (else the verdict came with the forward)
      LASER_TRY(accept_commit(nullptr, nullptr, logits, tokens, n_rows, B, m->cfg.vocab, &acc, n_accept, out_tokens, n_out,
                              g.stamps + STAMP_VERIFIED, stream));
    }
    LASER_CUDA(launch_overlapped(step_kernel, dim3(1), kStepThreads, 0, stream, g, 0, fused ? 1 : 0, n_rows, n_accept, out_tokens, n_out,
                                 host.report + tag % kSlots, tag));
    count_launch();
    return LASER_OK;
  };

  // A step emits at most Rs tokens of a sequence, so while a sequence has more than that to go for every step in flight, the
  // next step will be needed whatever those decide, and is queued without waiting for them; the device never idles between
  // steps.  A step that may not be needed (the last few, and all of them where an EOS token can end a text at any step) waits
  // for the report of the one before, while the device already drafts for it.  2-layer model, 4 sequences, 64 new tokens in 28
  // steps: 3.64 ms with a wait, two copies and four events after every step and ordinary launches of the small kernels, 2.38
  // without the waits and copies, 2.11 with the stage times taken by the kernels instead of by events between them.
  const int max_steps = p->max_new + 1;
  const unsigned tag0 = host.tag;
  int queued = 0, seen = 0, remaining = p->max_new, error = 0;
  LASER_TRY(queue_draft());
  while (remaining > 0 && error == 0 && (queued < max_steps || seen < queued)) {
    const int flight = queued - seen;
    if (flight > 0 && (queued == max_steps || p->eos_id >= 0 || flight >= kInFlight || remaining <= flight * Rs)) {
      unsigned long long r = 0;
      LASER_TRY(host.wait_report(tag0 + seen, stream, &r));
      remaining = int(r >> 32);
      error = int((r >> 24) & 0xffu);
      ++seen;
      continue;
    }
    LASER_TRY(queue_step(host.tag++, flight == 0 && queued > 0));
    ++queued;
    LASER_TRY(queue_draft());
  }
  if (error) LASER_TRY(laser_check(m, stream));   // a device-side error (capacity, a wait that ran out): reported, cleared
  LASER_CUDA(cudaMemcpyAsync(h, init, n_result * 4, cudaMemcpyDeviceToHost, stream));
  LASER_CUDA(cudaStreamSynchronize(stream));
  memcpy(out, h + at_out, size_t(B) * p->max_new * 4);
  memcpy(out_len, h + at_out_len, size_t(B) * 4);
  if (remaining > 0) { set_error("generation did not finish in %d steps", max_steps); return LASER_ERR_TIMEOUT; }
  if (stats) {
    unsigned long long count[COUNTERS];
    memcpy(count, h + at_counters, sizeof(count));
    float ms_prefill = 0;
    LASER_CUDA(cudaEventElapsedTime(&ms_prefill, host.begin, host.prefilled));
    stats->steps = int64_t(count[COUNT_STEPS]); stats->drafted = int64_t(count[COUNT_DRAFTED]);
    stats->accepted = int64_t(count[COUNT_ACCEPTED]); stats->emitted = int64_t(count[COUNT_EMITTED]);
    stats->launches = g_launches - launches0;
    stats->verify_calls = queued;
    stats->ms_prefill = ms_prefill; stats->ms_draft = float(1e-6 * double(count[NS_DRAFT]));
    stats->ms_verify = float(1e-6 * double(count[NS_VERIFY])); stats->ms_accept = float(1e-6 * double(count[NS_ACCEPT]));
    stats->ms_total = stats->ms_prefill + stats->ms_draft + stats->ms_verify + stats->ms_accept;
  }
  return LASER_OK;
}
