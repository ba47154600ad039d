// Causal attention of a prefill pass (Eq. 3): chunks of up to 32 prompt tokens against the paged bf16 KV cache, which already
// holds the keys and values of all of the pass's chunks.
//
// One CTA per (four consecutive chunks, head), a warp per chunk.  Consecutive chunks are mostly of one prompt, so a staged
// page serves 128 rows: the prompt's pages come two at a time through TMA (128-byte swizzle) into a ring of shared-memory
// stages, and every warp takes those that its rows see.  Where the four chunks are of several prompts the CTA takes the prompts
// one after another, and the warps of the others let a stage pass.  The first warp refills a stage once it has worked on the one
// behind it: a fifth warp for the copies would leave the four 168 registers a thread instead of 255, and they need more.
// A warp computes S = Q K^T and O += P V of 32 rows x 32 keys with warp-level MMA, so that a fragment of K or V feeds two row
// tiles, and the online softmax's shuffles and rescaling are paid once for 32 keys.
// Bound by latency - the chain from the score MMA through the softmax to the value MMA, with two warps a scheduler: tensor pipe 41 % busy, issue
// 35 %, shared memory 31 % - and by the CTAs that walk most keys (the host lists those first).  Head size 128 takes 255 registers,
// 4 bytes of which are spilled, so there is no room for more in flight.  The kernel for
// verify steps, which it replaces here, reads a fragment of K and V for 16 rows and takes a page's 16 keys at a time: 7B, prompts of 256 ..
// 1024 tokens, 61 us a layer for passes of 1024 rows; this one 107 us for passes of 2304 with the chunks as they come, 76 us with those
// that see most first.
#include "mma.cuh"
#include "model.cuh"
#include "tma.cuh"

namespace laser {
namespace {

using bf16 = __nv_bfloat16;
constexpr int kChunks = kPrefillShare;          // of a CTA: a warp each
constexpr int kRows = kPrefillChunk;            // of a chunk: two 16-row tiles
constexpr int kThreads = kChunks * 32;
constexpr int kStages = 4;
constexpr int kPages = 2;                       // of a stage: 32 keys

template <int DH>
struct Sizes {
  static constexpr int kHalves = DH / 64;                     // 64-element (128-byte) column blocks of a row
  static constexpr int kSub = 16 * 128;                       // bytes of 16 tokens x 64 elements
  static constexpr int kPage = 2 * kHalves * kSub;            // K then V
  static constexpr int kStage = kPages * kPage;
  static constexpr int kQRow = DH + 8;                        // padded row of the Q tile (elements)
  static constexpr int kSmem = 1024 + kStages * kStage + kChunks * kRows * kQRow * 2;
};

template <int DH>
__global__ void __launch_bounds__(kThreads, 2)
attn_prefill_kernel(const __grid_constant__ CUtensorMap kvmap, const bf16* q, const int32_t* __restrict__ seq_ids, const int32_t* row_ctx,
                    const int32_t* row_n, int n_chunks, int H, int Hkv, const int32_t* __restrict__ page_table, int pages_per_seq,
                    int layer_row0, bf16* __restrict__ out, int32_t* __restrict__ status) {
  using Z = Sizes<DH>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full_bar[kStages], empty_bar[kStages];
  __shared__ int s_keys[kChunks], s_seq[kChunks];   // keys that a chunk sees (0: it has no rows), its cache slot
  __shared__ int abort_flag;
  next_may_launch();
  const int c0 = blockIdx.y * kChunks, h = blockIdx.x, hk = h / (H / Hkv);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t raw = smem_u32(smem_raw), tiles = (raw + 1023u) & ~1023u;
  const uint32_t q_smem = tiles + kStages * Z::kStage;
  bf16* const q_ptr = reinterpret_cast<bf16*>(smem_raw + (tiles - raw) + kStages * Z::kStage);
  if (tid == 0) {
    abort_flag = 0;
    for (int s = 0; s < kStages; ++s) { mbar_init(smem_u32(&full_bar[s]), 1); mbar_init(smem_u32(&empty_bar[s]), kChunks); }
    mbar_fence_init();
    tma_prefetch_map(&kvmap);
  }
  wait_for_earlier();   // queries and the pass's own keys and values; what describes the rows
  if (tid < kChunks) {
    const int c = c0 + tid, n = c < n_chunks ? row_n[c] : 0;
    s_keys[tid] = n > 0 ? row_ctx[c] + n : 0;
    s_seq[tid] = n > 0 ? seq_ids[c] : -1;
  }
  __syncthreads();

  // Chunks first .. last - 1 are of one prompt, and see its first `keys` keys between them.
  auto next_prompt = [&](int& first, int& last, int& keys) {
    first = last;
    while (first < kChunks && s_keys[first] == 0) ++first;
    if (first == kChunks) return false;
    keys = 0;
    for (last = first; last < kChunks && (s_keys[last] == 0 || s_seq[last] == s_seq[first]); ++last) keys = max(keys, s_keys[last]);
    return true;
  };

  // The copies, by the first warp: where they are, and the next two pages.
  int put_first = 0, put_last = 0, put_keys = 0, put_k0 = 0, put_stage = 0, put_par = 1;   // (a fresh barrier passes a wait for the phase before its first)
  auto put = [&]() {          // false: a wait ran out
    if (put_k0 >= put_keys) {
      put_k0 = 0;
      if (!next_prompt(put_first, put_last, put_keys)) { put_keys = 0; return true; }
    }
    const bool free = mbar_wait_warp(smem_u32(&empty_bar[put_stage]), put_par, &abort_flag);
    if (free && lane == 0) {
      const int32_t* pt = page_table + size_t(s_seq[put_first]) * pages_per_seq;
      const uint32_t bar = smem_u32(&full_bar[put_stage]), dst = tiles + uint32_t(put_stage) * Z::kStage;
      mbar_expect_tx(bar, Z::kStage);
#pragma unroll
      for (int x = 0; x < kPages; ++x) {
        const int phys = pt[min((put_k0 >> 4) + x, (put_keys - 1) >> 4)];    // (past the last page: that one again, masked)
        const int rowk = layer_row0 + ((phys * 2) * Hkv + hk) * 16, rowv = layer_row0 + ((phys * 2 + 1) * Hkv + hk) * 16;
#pragma unroll
        for (int hf = 0; hf < Z::kHalves; ++hf) {
          tma_load_2d(dst + x * Z::kPage + hf * Z::kSub, &kvmap, hf * 64, rowk, bar);
          tma_load_2d(dst + x * Z::kPage + (Z::kHalves + hf) * Z::kSub, &kvmap, hf * 64, rowv, bar);
        }
      }
    }
    __syncwarp();
    put_k0 += 16 * kPages;
    if (++put_stage == kStages) { put_stage = 0; put_par ^= 1; }
    return free;
  };
  bool ok = true;
  if (warp == 0)
    for (int i = 0; i < kStages - 1; ++i) ok = ok && put();

  // ---- a chunk's warp ----
  const int c = c0 + warp;
  const int my_keys = s_keys[warp], nr = my_keys ? row_n[c] : 0, ctx = my_keys - nr;
  bf16* const my_q = q_ptr + warp * kRows * Z::kQRow;
  constexpr int kVec = DH / 8;                     // 16-byte pieces of a row
  {
    uint4 v[kRows * kVec / 32];
#pragma unroll
    for (int x = 0; x < kRows * kVec / 32; ++x) {
      const int i = x * 32 + lane, r = i / kVec, d = i % kVec * 8;
      v[x] = r < nr ? *reinterpret_cast<const uint4*>(q + (size_t(c) * kRows + r) * H * DH + size_t(h) * DH + d) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int x = 0; x < kRows * kVec / 32; ++x) {
      const int i = x * 32 + lane, r = i / kVec, d = i % kVec * 8;
      *reinterpret_cast<uint4*>(my_q + r * Z::kQRow + d) = v[x];
    }
  }
  __syncwarp();
  const int g = lane >> 2, qd = lane & 3, mat = lane >> 3;
  const float sl2 = rsqrtf(float(DH)) * 1.4426950408889634f;
  const uint32_t q_frag = q_smem + uint32_t((warp * kRows + (lane & 7) + (mat & 1) * 8) * Z::kQRow + (mat >> 1) * 8) * 2;
  float o[2][DH / 8][4];
#pragma unroll
  for (int t = 0; t < 2; ++t)
#pragma unroll
    for (int j = 0; j < DH / 8; ++j) o[t][j][0] = o[t][j][1] = o[t][j][2] = o[t][j][3] = 0.f;
  // rows g and g + 8 of each tile: running max and sum
  float m_run[2][2] = {{-INFINITY, -INFINITY}, {-INFINITY, -INFINITY}}, l_run[2][2] = {};

  int stage = 0, par = 0;
  for (int first = 0, last = 0, keys; ok && next_prompt(first, last, keys);) {
    const bool mine = warp >= first && warp < last;
    for (int k0 = 0; k0 < keys; k0 += 16 * kPages) {
      const int s = stage;
      if (warp == 0) ok = put();
      ok = ok && mbar_wait_warp(smem_u32(&full_bar[s]), par, &abort_flag);
      if (!ok) break;
      if (++stage == kStages) { stage = 0; par ^= 1; }
      if (mine && k0 < my_keys) {
        const uint32_t base = tiles + uint32_t(s) * Z::kStage;
        float sc[2][4][4];     // [row tile][eight keys]
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
          for (int n = 0; n < 4; ++n) sc[t][n][0] = sc[t][n][1] = sc[t][n][2] = sc[t][n][3] = 0.f;
        {
          const int key = (lane & 7) + (mat >> 1) * 8;
#pragma unroll
          for (int ks = 0; ks < DH / 16; ++ks) {
            const int col = (ks & 3) * 2 + (mat & 1);
            uint32_t qa[2][4], kb[4];
            ldsm_x4(qa[0], q_frag + ks * 32);
            ldsm_x4(qa[1], q_frag + 16 * Z::kQRow * 2 + ks * 32);
#pragma unroll
            for (int x = 0; x < kPages; ++x) {
              ldsm_x4(kb, base + x * Z::kPage + (ks >> 2) * Z::kSub + key * 128 + ((col ^ (key & 7)) << 4));
#pragma unroll
              for (int t = 0; t < 2; ++t) {
                mma16816(sc[t][2 * x], qa[t], kb[0], kb[1]);
                mma16816(sc[t][2 * x + 1], qa[t], kb[2], kb[3]);
              }
            }
          }
        }
        // a row sees the keys up to itself (rows past the chunk's end copy its last)
        if (k0 + 16 * kPages > ctx + 1) {
#pragma unroll
          for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int n = 0; n < 4; ++n)
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (k0 + n * 8 + 2 * qd + (e & 1) > ctx + min(t * 16 + g + (e >> 1) * 8, nr - 1)) sc[t][n][e] = -INFINITY;
        }
        uint32_t pf[2][kPages][4];
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
          for (int r = 0; r < 2; ++r) {        // row g + 8 r of the tile
            float mx = m_run[t][r];
#pragma unroll
            for (int n = 0; n < 4; ++n) mx = fmaxf(mx, fmaxf(sc[t][n][2 * r], sc[t][n][2 * r + 1]));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float mu = mx == -INFINITY ? 0.f : mx, al = exp2f((m_run[t][r] - mu) * sl2);
            m_run[t][r] = mx;
            float sum = 0.f;
#pragma unroll
            for (int n = 0; n < 4; ++n) {
              const float p0 = exp2f((sc[t][n][2 * r] - mu) * sl2), p1 = exp2f((sc[t][n][2 * r + 1] - mu) * sl2);
              sum += p0 + p1;
              pf[t][n >> 1][(n & 1) * 2 + r] = pack_bf16(p0, p1);
            }
            l_run[t][r] = l_run[t][r] * al + sum;
#pragma unroll
            for (int j = 0; j < DH / 8; ++j) { o[t][j][2 * r] *= al; o[t][j][2 * r + 1] *= al; }
          }
        {
          const int key = (lane & 7) + (mat & 1) * 8;
#pragma unroll
          for (int j = 0; j < DH / 16; ++j) {
            const int col = (j & 3) * 2 + (mat >> 1);
#pragma unroll
            for (int x = 0; x < kPages; ++x) {
              uint32_t vb[4];
              ldsm_x4_t(vb, base + x * Z::kPage + (Z::kHalves + (j >> 2)) * Z::kSub + key * 128 + ((col ^ (key & 7)) << 4));
#pragma unroll
              for (int t = 0; t < 2; ++t) {
                mma16816(o[t][2 * j], pf[t][x], vb[0], vb[1]);
                mma16816(o[t][2 * j + 1], pf[t][x], vb[2], vb[3]);
              }
            }
          }
        }
        __syncwarp();
      }
      if (lane == 0) mbar_arrive(smem_u32(&empty_bar[s]));
    }
  }
  // (after a wait that ran out: copies in flight land within microseconds)
  if (!ok) { const long long t0 = clock64(); while (clock64() - t0 < 2000000) {} }

  // ---- the rows' results (zeros where a chunk has no row) ----
  if (c < n_chunks) {
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float l = l_run[t][r];
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        const int row = t * 16 + g + r * 8;
        const float inv = row < nr && l > 0.f && ok ? 1.f / l : 0.f;
        bf16* dst = out + (size_t(c) * kRows + row) * H * DH + size_t(h) * DH + 2 * qd;
#pragma unroll
        for (int j = 0; j < DH / 8; ++j)
          *reinterpret_cast<uint32_t*>(dst + j * 8) = pack_bf16(o[t][j][2 * r] * inv, o[t][j][2 * r + 1] * inv);
      }
  }
  if (lane == 0 && abort_flag) atomicCAS(status, 0, LASER_ERR_TIMEOUT);
}

}  // namespace

laser_status attention_prefill_launch(laser_model* m, laser_kv* kv, int layer, const int32_t* seq_ids, int n_chunks, cudaStream_t stream) {
  const int H = m->cfg.n_heads, Hkv = m->cfg.n_kv_heads;
  const int layer_row0 = int(int64_t(kv->n_pages) * 2 * Hkv * 16 * layer);
  auto launch = [&](auto kernel, int smem) -> laser_status {
    LASER_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    LASER_CUDA(launch_overlapped(kernel, dim3(unsigned(H), unsigned(ceil_div(n_chunks, kChunks))), kThreads, size_t(smem), stream, kv->pages_map,
                                 m->q, seq_ids, m->row_ctx, m->row_n, n_chunks, H, Hkv, kv->page_table, kv->pages_per_seq, layer_row0,
                                 m->attn, m->status));
    return LASER_OK;
  };
  LASER_TRY(m->cfg.head_dim == 128 ? launch(attn_prefill_kernel<128>, Sizes<128>::kSmem) : launch(attn_prefill_kernel<64>, Sizes<64>::kSmem));
  count_launch();
  return LASER_OK;
}

}  // namespace laser
