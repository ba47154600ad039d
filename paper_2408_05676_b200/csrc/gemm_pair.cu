// Dense contractions of the verify forward for many token rows: the same acc[r][n] = sum_k A[r][k] * W[n][k] and
// the same fused epilogues as gemm.cu, for steps whose row count makes the tensor pipe and the L2->SM traffic the
// bound instead of the weight stream.
//
// A pair of CTAs (a cluster of two, one CTA per SM) runs 256-row MMAs together (cta_group::2): each CTA stages 128
// of the tile's weight rows and half of its token rows, so a K block of a 256 x NT tile costs an SM 16 KB + NT/2 x
// 128 B instead of 16 KB + NT x 128 B.  The kernel is persistent: pair p walks the tiles p, p + P, .., and two
// accumulators in tensor memory let the epilogue of one tile run under the main loop of the next.  The tiles left
// over after the last full wave are cut along K over all pairs where that pays; the pairs that share a tile exchange
// fp32 partial sums through a scratch in L2 and each finishes a slice of its token rows, in a fixed order of summation.
// How a tile is cut follows from its weight tile alone: all token tiles of a weight tile are whole, or all are cut at the
// same K blocks.  A row's result then does not depend on its place in the step, so that a token among drafts gets the
// logits that it gets alone (and results are the same from run to run).
//   warps 0, 10  TMA producers of the CTA's own halves (weights, activations); completion bytes count on the pair's
//              first CTA
//   warp 1     MMA issuer (first CTA only); commits free the stages of both CTAs
//   warps 2-9  epilogue, two groups of four warps on alternate chunks of 32 token rows: tensor memory -> staging
//              buffer -> one warp per token row
// One CTA per SM holds more than half of the shared memory, so no other kernel's tensor-memory user is ever resident
// beside it: the pair allocation cannot meet a foreign or a half-made allocation on one of its two SMs.
// What bounds it: the tensor pipe in the main loop (192-row tiles: 0.265 us a K block and pair = 1.75 PFLOP/s at 1.85 GHz;
// long steps settle at the power cap) and, around it, about 2.5 us from the previous kernel's end to the first MMA and the
// last tile's epilogue.  Against the form it replaced (two 128-row weight tiles a CTA, one CTA per SM, single-CTA MMAs; A/B):
// 7B step of 64 sequences x 9 rows 12.34 -> 10.77 ms, tree step of 16 x 17 rows 7.34 -> 6.39, precise mode 16 x 9 rows 7.02 ->
// 6.26, 13B layers with 64 x 17 rows 8.11 -> 6.98.  Two accumulators of 256 rows each beat both 512-row tiles (weights or
// tokens), whose epilogue nothing overlaps.
// Every wait is bounded, as in gemm.cu.
#include <algorithm>
#include <type_traits>

#include "epilogue.cuh"
#include "gemm_pair.cuh"
#include "tma.cuh"
#include "umma.cuh"

namespace laser {
namespace {

constexpr int kPairThreads = 352;
constexpr int kEpiWarps = 8;
constexpr int kMaxStages = 8;
constexpr int kChunk = 32;                       // token rows in a group's staging buffer
constexpr int kStgRow = 132;                     // floats per staged row
constexpr int kStgBytes = kChunk * kStgRow * 4;  // 16.5 KB per group
constexpr int kPairSmem = 220 * 1024;   // + up to 6.2 KB of static shared memory

struct PairPlan {
  int N, NT, n_tt, KB, stages;
  int P;                        // pairs in the grid
  int full_tiles, rem_tiles;    // whole tiles; tiles cut along K: every token tile of the last weight tiles
  int S, k;                     // cut tiles: K ranges of a tile, K blocks of a range
  int peer_cycles;              // how long a contributor waits for the others of its tile
  float* scratch;               // [pair][rank][NT][128 features]
  int32_t* state;               // [cut tile][rank][kPairState]
};

struct Item { int tile, kb0, kb1, C, c; };   // C contributors, this pair is number c

// A pair's whole tiles, then at most one range of a cut tile.
__device__ __forceinline__ bool get_item(const PairPlan& pl, int p, int idx, Item& it) {
  const int n_whole = pl.full_tiles > p ? (pl.full_tiles - 1 - p) / pl.P + 1 : 0;
  if (idx < n_whole) {
    it.tile = p + idx * pl.P; it.kb0 = 0; it.kb1 = pl.KB; it.C = 1; it.c = 0;
    return true;
  }
  if (idx > n_whole || p >= pl.rem_tiles * pl.S) return false;
  const int i = p / pl.S;
  it.tile = pl.full_tiles + i; it.C = pl.S; it.c = p - i * pl.S;
  it.kb0 = it.c * pl.k;
  it.kb1 = min(pl.KB, it.kb0 + pl.k);
  return true;
}

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t local_addr, uint32_t rank) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local_addr), "r"(rank));
  return remote;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// bounded wait on a barrier that the other CTA of the pair arrives on as well
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  const long long t0 = clock64();
  for (;;) {
    for (int i = 0; i < 256; ++i) {
      uint32_t ok;
      asm volatile("{\n.reg .pred p;\nmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                   : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
      if (ok) return true;
    }
    if (*abort_flag) return false;
    if (clock64() - t0 > kWaitCycles) { *abort_flag = 1; return false; }
  }
}
__device__ __forceinline__ void st_shared_f32(uint32_t addr, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ float4 ld_shared_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void epi_barrier() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void group_barrier(int group) { asm volatile("bar.sync %0, 128;" ::"r"(2 + group) : "memory"); }

// A tile is 256 weight rows x NT token rows; tensor memory holds two accumulators of them.
// PARTS = 2: activations as hi + lo bf16 pairs, both multiplied with the staged weight block into one accumulator.
template <int EPI, int PARTS>
__global__ void __launch_bounds__(kPairThreads, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmA, const GemmEpilogue e,
                 const PairPlan pl, int32_t* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], acc_full[2], acc_empty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag, s_last, s_go;
  __shared__ float s_rstd[256];
  __shared__ int s_pos[256], s_page[256];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int NT = pl.NT, stages = pl.stages;
  const uint32_t tiles = (smem_u32(smem_raw) + 1023u) & ~1023u;
  constexpr uint32_t w_bytes = kBM * 128;
  const uint32_t a_bytes = uint32_t(NT / 2) * 128, stage_bytes = w_bytes + PARTS * a_bytes;
  const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // (uniform)
  const int p = blockIdx.x >> 1, rank = blockIdx.x & 1;

  if (threadIdx.x == 0) {
    tma_prefetch_map(&tmW);
    tma_prefetch_map(&tmA);
    abort_flag = 0;
    for (int s = 0; s < stages; ++s) { mbar_init(smem_u32(&full_bar[s]), 1); mbar_init(smem_u32(&empty_bar[s]), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&acc_full[b]), 1); mbar_init(smem_u32(&acc_empty[b]), 2 * kEpiWarps); }
    mbar_fence_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  Item it;
  bool more = get_item(pl, p, 0, it);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync_all();   // the peer signals this CTA's barriers
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
  const uint32_t elected = elect_one();

  if (warp == 0 || warp == 10) {
    {
      // ---- TMA producers: warp 0 the weight tiles, warp 10 the activation tiles ----
      // A K block is due every 0.2 to 0.6 us, so these loops hold everything that changes only with the
      // tile in registers (a division per K block was enough to pace the kernel: 0.41 us).
      const bool act = warp == 10;
      const uint32_t full0 = map_to_rank(smem_u32(&full_bar[0]), 0), full_own = smem_u32(&full_bar[0]), empty0 = smem_u32(&empty_bar[0]);
      const uint64_t policy = act ? make_policy_evict_last() : make_policy_evict_first();
      int s = 0, par = 1, idx = 0, n = 0;    // (a fresh barrier passes a wait for the phase before its first)
      bool ok = true;
      if (act) asm volatile("griddepcontrol.wait;" ::: "memory");   // the weights depend on no earlier kernel
      for (; ok && more; more = get_item(pl, p, ++idx, it)) {
        const int wt = it.tile / pl.n_tt;
        const int T = wt * 2 + rank, r0 = (it.tile - wt * pl.n_tt) * NT + rank * (NT / 2);
        for (int kb = it.kb0; kb < it.kb1; ++kb, ++n) {
          ok = mbar_wait_hot(empty0 + uint32_t(s) * 8, par, &abort_flag);
          if (!ok) break;
          const uint32_t bar = full0 + uint32_t(s) * 8, dst = tiles + uint32_t(s) * stage_bytes;
          if (act) {
#pragma unroll
            for (int q = 0; q < PARTS; ++q)
              tma_load_2d_pair(dst + w_bytes + uint32_t(q) * a_bytes, &tmA, (q ? e.a_lo_off : 0) + kb * kBK, r0, bar, policy, elected);
          } else {
            if (rank == 0 && elected) mbar_expect_tx(full_own + uint32_t(s) * 8, 2 * stage_bytes);
            if (EPI == EPI_SWIGLU) {   // 64 gate rows and the 64 up rows of the same features
              tma_load_2d_pair(dst, &tmW, kb * kBK, T * 64, bar, policy, elected);
              tma_load_2d_pair(dst + w_bytes / 2, &tmW, kb * kBK, e.f + T * 64, bar, policy, elected);
            } else {
              tma_load_2d_pair(dst, &tmW, kb * kBK, T * kBM, bar, policy, elected);
            }
          }
          if (++s == stages) { s = 0; par ^= 1; }
        }
      }
      // the commits on this CTA's barriers must have landed before it may exit: the slots in the order of their last
      // use, from s when the ring has been full, from 0 otherwise
      if (!act)
        for (int i = min(n, stages); i > 0 && ok; --i) {
          if (n < stages) { ok = mbar_wait(empty0 + uint32_t(n - i) * 8, 0, &abort_flag); continue; }
          ok = mbar_wait(empty0 + uint32_t(s) * 8, par, &abort_flag);
          if (++s == stages) { s = 0; par ^= 1; }
        }
      if (!ok) { const long long t0 = clock64(); while (clock64() - t0 < 2000000) {} }   // copies in flight land within microseconds
    }
  } else if (warp == 1) {
    if (rank == 0) {  // ---- MMA issuer ----
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(NT >> 3) << 17) | (uint32_t(256 >> 4) << 24);
      bool ok = true;
      const uint64_t wdesc0 = umma_desc(tiles);
      int s = 0, par = 0;
      for (int idx = 0; ok && more; more = get_item(pl, p, ++idx, it)) {
        const int buf = idx & 1;
        const uint32_t acc = tmem + uint32_t(buf) * 256;
        ok = mbar_wait_cluster(smem_u32(&acc_empty[buf]), ((idx >> 1) & 1) ^ 1, &abort_flag);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t accumulate = 0;
        for (int kb = it.kb0; kb < it.kb1 && ok; ++kb) {
          ok = mbar_wait_hot(smem_u32(&full_bar[s]), par, &abort_flag);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t stage = wdesc0 + uint64_t(uint32_t(s) * (stage_bytes >> 4));
#pragma unroll
          for (int q = 0; q < PARTS; ++q)
            umma_kblock_pair(acc, stage, stage + uint64_t((w_bytes >> 4) + uint32_t(q) * (a_bytes >> 4)), idesc, accumulate | uint32_t(q), elected);
          accumulate = 1;
          umma_commit_pair(smem_u32(&empty_bar[s]), 3, elected);
          if (++s == stages) { s = 0; par ^= 1; }
        }
        umma_commit_pair(smem_u32(&acc_full[buf]), 3, elected);
      }
    }
  } else {
    // ---- epilogue ----
    const int et = threadIdx.x - 64, group = (warp - 2) >> 2, quarter = warp & 3;
    const uint32_t stg = tiles + uint32_t(stages) * stage_bytes + uint32_t(group) * kStgBytes;
    const uint32_t stg_w = stg + uint32_t(quarter * 32 + lane) * 4;
    const uint32_t lanes = uint32_t(quarter * 32) << 16;
    const uint32_t lead_empty0 = map_to_rank(smem_u32(&acc_empty[0]), 0);
    asm volatile("griddepcontrol.wait;" ::: "memory");   // what follows reads earlier kernels' results
    int ctx_r0 = -1;
    auto row_context = [&](int r0) {   // per-row scale and cache coordinates of the tile's token rows
      if (r0 == ctx_r0) return;
      ctx_r0 = r0;
      epi_barrier();
      for (int j = et; j < NT; j += 256) {
        const int r = r0 + j;
        float rstd = 1.f;
        int pos = -1, page = 0;
        if (r < e.R_rows) {
          if (e.sumsq_in) {
            float ss = 0.f;
#pragma unroll 16
            for (int tt = 0; tt < e.sumsq_in_tiles; ++tt) ss += e.sumsq_in[size_t(tt) * e.sumsq_ld + r];
            rstd = rsqrtf(ss * e.inv_d + e.eps);
          }
          if (EPI == EPI_VERDICT) pos = r < e.R_store ? e.row_draft[r] : -1;
          if (EPI == EPI_QKV) {
            pos = e.row_pos[r];
            if (pos >= 0) page = e.page_table[size_t(e.row_seq[r]) * e.pages_per_seq + (pos >> 4)];
          }
        }
        s_rstd[j] = rstd; s_pos[j] = pos; s_page[j] = page;
      }
      epi_barrier();
    };
    // Operands of the token rows r .. r + CNT - 1 of weight tile wt that the epilogue reads from global memory, one
    // 16-byte load per row and lane: the residual's four features, or half of the eight rotary values that the lane and
    // its rotation partner both need.  They are requested a chunk ahead: an L2 round trip (about 1 us here) costs as much
    // as the rest of a chunk.
    auto fetch_rows = [&](int r, int wt, auto& g) {
      constexpr int CNT = sizeof(g) / sizeof(float4);
      if (EPI != EPI_RESID && EPI != EPI_QKV) return;
      const LaneCtx lc = make_lane_ctx<EPI>(e, wt * kBM, lane, pl.N);
#pragma unroll
      for (int x = 0; x < CNT; ++x) {
        g[x] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r + x < e.R_rows && lc.in_range) {
          if (EPI == EPI_RESID) g[x] = __ldcg(reinterpret_cast<const float4*>(e.resid + size_t(r + x) * pl.N + lc.n));
          if (EPI == EPI_QKV && lc.kind < 2)   // c0 s0 c1 s1 in the first half of the head, c2 s2 c3 s3 in the second
            g[x] = __ldg(reinterpret_cast<const float4*>(e.rope + size_t(r + x) * e.dh + lc.rope_off + (lc.sg < 0.f ? 0 : 4)));
        }
      }
    };
    // a warp finishes the token rows from row j0 of the tile (row r0 + j0 of the step) on; acc_of(x): the lane's four
    // features of the x-th
    auto finish_rows = [&](int r0, int wt, int j0, const auto& g, auto&& acc_of) {
      constexpr int CNT = sizeof(g) / sizeof(float4);
      const int n0 = wt * kBM;
      const LaneCtx lc = make_lane_ctx<EPI>(e, n0, lane, pl.N);
      uint2 gain4 = make_uint2(0u, 0u);
      if (EPI == EPI_RESID && lc.in_range) gain4 = *reinterpret_cast<const uint2*>(e.gain_next + lc.n);
#pragma unroll
      for (int x = 0; x < CNT; ++x) {
        const int j = j0 + x, r = r0 + j;
        const float4 acc = acc_of(x);
        const bool live = r < e.R_rows && !abort_flag;
        const float rstd = s_rstd[j];
        if (EPI == EPI_PLAIN) epi_plain(e, lc, r, live, acc, rstd, pl.N);
        else if (EPI == EPI_VERDICT) epi_verdict(e, lc, r, live, lane, acc, rstd, pl.N, wt, s_pos[j]);
        else if (EPI == EPI_RESID) epi_resid(e, lc, r, live, lane, acc, pl.N, wt, g[x], gain4);
        else if (EPI == EPI_SWIGLU) epi_swiglu(e, r, live, wt * 64, lane, acc, rstd);
        else {
          float4 o;
          o.x = __shfl_xor_sync(0xffffffffu, g[x].x, lc.shift); o.y = __shfl_xor_sync(0xffffffffu, g[x].y, lc.shift);
          o.z = __shfl_xor_sync(0xffffffffu, g[x].z, lc.shift); o.w = __shfl_xor_sync(0xffffffffu, g[x].w, lc.shift);
          const bool low = lc.sg < 0.f;
          epi_qkv(e, lc, r, live, acc, rstd, s_pos[j], s_page[j], low ? g[x] : o, low ? o : g[x]);
        }
      }
    };
    auto tile_state = [&](const Item& it) { return pl.state + ((it.tile - pl.full_tiles) * 2 + rank) * kPairState; };
    auto tile_valid = [&](int wt) { return EPI == EPI_SWIGLU ? wt * 64 < e.f : wt * kBM < pl.N; };
    // (after a wait that ran out the loops go on, without storing: every warp still meets every barrier)
    int idx = 0;
    for (; more; more = get_item(pl, p, ++idx, it)) {
      const int buf = idx & 1, wt = (it.tile / pl.n_tt) * 2 + rank, r0 = (it.tile % pl.n_tt) * NT;
      const bool finish = it.C == 1 && tile_valid(wt), publish = it.C > 1;
      row_context(r0);
      float4 g[8];
      if (finish && group * kChunk < NT) fetch_rows(r0 + group * kChunk + quarter * 8, wt, g);
      mbar_wait(smem_u32(&acc_full[buf]), (idx >> 1) & 1, &abort_flag);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // tensor memory -> staging buffer -> rows: finished, or (cut tile) published as partial sums
      if (finish || publish) {
        const uint32_t src = tmem + uint32_t(buf) * 256 + lanes;
        float* part = pl.scratch + (size_t(p) * 2 + rank) * NT * kBM + 4 * lane;
        for (int ch = group; ch * kChunk < NT; ch += 2) {
          uint32_t v0[16], v1[16];
          tmem_ld16(src + uint32_t(ch * kChunk), v0);
          tmem_ld16(src + uint32_t(ch * kChunk + 16), v1);   // past NT: still inside this accumulator's columns
          tmem_ld_wait();
          group_barrier(group);   // the group is done with the chunk before
#pragma unroll
          for (int x = 0; x < 16; ++x) {
            st_shared_f32(stg_w + uint32_t(x) * (kStgRow * 4), __uint_as_float(v0[x]));
            st_shared_f32(stg_w + uint32_t(16 + x) * (kStgRow * 4), __uint_as_float(v1[x]));
          }
          float4 gn[8];
          if (finish && (ch + 2) * kChunk < NT) fetch_rows(r0 + (ch + 2) * kChunk + quarter * 8, wt, gn);
          group_barrier(group);   // the chunk is staged
          const int j0 = ch * kChunk + quarter * 8;
          if (j0 < NT) {          // (rows past NT belong to the next token tile)
            auto staged = [&](int x) { return ld_shared_f4(stg + uint32_t((quarter * 8 + x) * kStgRow + 4 * lane) * 4); };
            if (finish) {
              finish_rows(r0, wt, j0, g, staged);
            } else {
#pragma unroll
              for (int x = 0; x < 8; ++x) __stcg(reinterpret_cast<float4*>(part + size_t(j0 + x) * kBM), staged(x));
            }
          }
#pragma unroll
          for (int x = 0; x < 8; ++x) g[x] = gn[x];
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(lead_empty0 + uint32_t(buf) * 8);
      if (publish) {
        epi_barrier();
        if (et == 0) {
          __threadfence();
          s_last = atomicAdd(tile_state(it), 1) == it.C - 1;
        }
      }
    }
    // A cut tile (a pair's last item): each contributor sums and finishes a slice of the token rows, after its partial sums
    // are published.  It waits for its peers only so long: they may not be running, if other kernels hold their SMs.
    // A slice given up is marked, and the contributor that arrives last takes it over; between the mark and the arrival
    // count each side writes its own before it reads the other's, and a compare-and-swap settles who goes on.
    if (idx > 0 && get_item(pl, p, idx - 1, it) && it.C > 1) {
      const int wt = (it.tile / pl.n_tt) * 2 + rank, r0 = (it.tile % pl.n_tt) * NT;
      row_context(r0);
      const int first = p - it.c;
      int32_t* state = tile_state(it);             // arrived, slices finished, one mark per slice
      const int sl = (NT / 4 + it.C - 1) / it.C;   // rows of a slice, in units of four
      // RB rows x all contributors' partial sums of a warp are requested together: one L2 round trip per batch
      auto sum_rows = [&](int j, auto rb_tag, auto cb_tag) {
        constexpr int RB = decltype(rb_tag)::value, CB = decltype(cb_tag)::value;
        const int q1 = min(NT, (j + 1) * sl * 4);
        for (int q = j * sl * 4 + (warp - 2) * RB; q < q1; q += kEpiWarps * RB) {
          float4 g[RB], sum[RB];
          fetch_rows(r0 + q, wt, g);
#pragma unroll
          for (int x = 0; x < RB; ++x) sum[x] = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int cb = 0; cb < it.C; cb += CB) {
            float4 v[CB][RB];
#pragma unroll
            for (int c = 0; c < CB; ++c) {
              const int pair = first + min(cb + c, it.C - 1);
              const float* b = pl.scratch + ((size_t(pair) * 2 + rank) * NT + q) * kBM + 4 * lane;
#pragma unroll
              for (int x = 0; x < RB; ++x)
                v[c][x] = cb + c < it.C ? __ldcg(reinterpret_cast<const float4*>(b + size_t(x) * kBM)) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int c = 0; c < CB; ++c)
#pragma unroll
              for (int x = 0; x < RB; ++x) { sum[x].x += v[c][x].x; sum[x].y += v[c][x].y; sum[x].z += v[c][x].z; sum[x].w += v[c][x].w; }
          }
          if (tile_valid(wt)) finish_rows(r0, wt, q, g, [&](int x) { return sum[x]; });
        }
      };
      auto finish_slice = [&](int j) {
        if (it.C == 2) sum_rows(j, std::integral_constant<int, 8>{}, std::integral_constant<int, 2>{});
        else if (it.C <= 4) sum_rows(j, std::integral_constant<int, 4>{}, std::integral_constant<int, 4>{});
        else sum_rows(j, std::integral_constant<int, 2>{}, std::integral_constant<int, 8>{});
        epi_barrier();
        if (et == 0 && atomicAdd(state + 1, 1) == it.C - 1)   // the tile's last slice: ready for the next launch
          for (int x = 0; x < it.C + 2; ++x) atomicExch(state + x, 0);
      };
      if (et == 0) {
        const long long t0 = clock64();
        int have = 0;
        do asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(have) : "l"(state) : "memory");
        while (have < it.C && clock64() - t0 < pl.peer_cycles);
        bool mine = have >= it.C;
        if (!mine) {
          atomicExch(state + 2 + it.c, 1);
          __threadfence();
          mine = atomicAdd(state, 0) >= it.C && atomicCAS(state + 2 + it.c, 1, 2) == 1;
          __threadfence();
        }
        s_go = mine;
      }
      epi_barrier();
      const bool last = s_last, mine = s_go;
      if (mine) finish_slice(it.c);
      if (last) {
        for (int j = 0; j < it.C; ++j) {
          if (j == it.c) continue;
          epi_barrier();
          if (et == 0) {
            __threadfence();
            s_go = atomicAdd(state + 2 + j, 0) == 1 && atomicCAS(state + 2 + j, 1, 2) == 1;
            __threadfence();
          }
          epi_barrier();
          if (s_go) finish_slice(j);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
  if (threadIdx.x == 0 && abort_flag) atomicCAS(status, 0, LASER_ERR_TIMEOUT);
}

// a cluster of two, and programmatic dependent launch as in gemm.cu
cudaLaunchConfig_t pair_config(cudaLaunchAttribute (&attr)[2], cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * kPairCount, 1, 1);
  cfg.blockDim = dim3(kPairThreads, 1, 1);
  cfg.dynamicSmemBytes = kPairSmem;    // all of it, whatever the stages take: one CTA per SM
  cfg.stream = stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

template <int EPI, int PARTS>
laser_status launch_parts(const CUtensorMap& tw, const CUtensorMap& ta, const GemmEpilogue& e, const PairPlan& pl, int32_t* status,
                          cudaStream_t stream) {
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = pair_config(attr, stream);
  LASER_CUDA(cudaFuncSetAttribute(gemm_pair_kernel<EPI, PARTS>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem));
  LASER_CUDA(cudaLaunchKernelEx(&cfg, gemm_pair_kernel<EPI, PARTS>, tw, ta, e, pl, status));
  return LASER_OK;
}

template <int EPI>
laser_status launch(const CUtensorMap& tw, const CUtensorMap& ta, const GemmEpilogue& e, const PairPlan& pl, int32_t* status,
                    cudaStream_t stream) {
  return e.a_lo_off ? launch_parts<EPI, 2>(tw, ta, e, pl, status, stream) : launch_parts<EPI, 1>(tw, ta, e, pl, status, stream);
}

int stage_count(int NT, int parts) {
  return std::min(kMaxStages, (kPairSmem - 1024 - 2 * kStgBytes) / (kBM * 128 + parts * (NT / 2) * 128));
}

// The tiles of a launch: whole ones in full waves, and the rest cut, from a weight tile's first token tile on.  Every cut
// tile has at least two pairs, which take one range each (no cut where the rest fills more than half of the pairs).
struct Cut { int full_tiles, rem_tiles, S, k; };
Cut cut_of(int tiles, int n_tt, int KB, bool split) {
  Cut c{tiles, 0, 1, KB};
  const int full = tiles / kPairCount * kPairCount / n_tt * n_tt, rem = tiles - full;
  if (!split || rem == 0 || 2 * rem > kPairCount) return c;
  c.full_tiles = full; c.rem_tiles = rem;
  c.k = ceil_div(KB, kPairCount / rem);
  c.S = ceil_div(KB, c.k);
  return c;
}

}  // namespace

size_t gemm_pair_scratch_floats(int R_pad) { return size_t(kPairCount) * 2 * std::min(R_pad, 256) * kBM; }

GemmPairShape gemm_pair_shape(int R_pad, int N, int K, int epi, bool pairs) {
  const int parts = pairs ? 2 : 1, KB = ceil_div(K, kBK);
  const int w256 = ceil_div(epi == EPI_SWIGLU ? ceil_div(N / 2, 64) : ceil_div(N, kBM), 2);   // 256-row weight tiles
  GemmPairShape best{};
  best.us = 1e30;
  const int least = ceil_div(R_pad, 256);
  for (int n_tt = least; n_tt <= least + 3; ++n_tt) {
    const int NT = ceil_div(ceil_div(R_pad, n_tt), 16) * 16;
    if ((n_tt - 1) * NT >= R_pad) continue;   // the last tile would be empty
    const int tiles = w256 * n_tt;
    // Constants fitted on the 7B and 13B layer shapes at 16 .. 2048 rows, each launch varied alone inside the step.  A K
    // block's MMAs take 1.2 ns per token row (1.75 PFLOP/s while the clock holds); below about 100 rows its 16 KB of
    // weights per SM take 0.16 us.  A cut tile costs 7 us of exchange; a launch ends with the last tile's epilogue, NT / 40 us.
    const double kb_us = std::max(0.16, 0.035 + 0.0012 * NT * parts);
    auto wave_us = [&](int wave_tiles, int kbs) {   // its distinct weight tiles come from HBM
      const double fresh = std::min(double(w256), double(wave_tiles) / n_tt);
      return std::max(kbs * kb_us, fresh * KB * (256 * kBK * 2) / 6.1e6);
    };
    for (int split = 0; split < 2; ++split) {
      const Cut cut = cut_of(tiles, n_tt, KB, split != 0);
      if (split && cut.rem_tiles == 0) continue;
      const int waves = split ? ceil_div(cut.full_tiles, kPairCount) : tiles / kPairCount;
      double us = NT / 40.0 + waves * wave_us(kPairCount, KB);
      if (split) us += wave_us(cut.rem_tiles, cut.k) + 7.0;
      else if (tiles % kPairCount) us += wave_us(tiles % kPairCount, KB);
      if (us < best.us) best = GemmPairShape{NT, n_tt, split, us};
    }
  }
  return best;
}

bool gemm_pair_fits() {
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = pair_config(attr, nullptr);
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaFuncSetAttribute(gemm_pair_kernel<EPI_QKV, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&clusters, gemm_pair_kernel<EPI_QKV, 1>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return clusters >= kPairCount;
}

laser_status gemm_pair_launch(laser_model* m, const GemmPairShape& sh, const CUtensorMap& tw, const CUtensorMap& ta, int N, int K, int epi,
                              const GemmEpilogue& e, cudaStream_t stream) {
  PairPlan pl = {};
  pl.N = N;
  pl.NT = sh.NT;
  pl.n_tt = sh.n_tt;
  pl.KB = ceil_div(K, kBK);
  pl.stages = stage_count(sh.NT, e.a_lo_off ? 2 : 1);
  pl.P = kPairCount;
  const int w256 = ceil_div(epi == EPI_SWIGLU ? ceil_div(N / 2, 64) : ceil_div(N, kBM), 2);
  const int tiles = w256 * pl.n_tt;
  const Cut cut = cut_of(tiles, pl.n_tt, pl.KB, sh.split != 0);
  pl.full_tiles = cut.full_tiles; pl.rem_tiles = cut.rem_tiles;
  pl.S = cut.S; pl.k = cut.k;
  pl.peer_cycles = m->peer_cycles;
  pl.scratch = m->pair_scratch;
  pl.state = m->pair_state;
  switch (epi) {
    case EPI_PLAIN: return launch<EPI_PLAIN>(tw, ta, e, pl, m->status, stream);
    case EPI_RESID: return launch<EPI_RESID>(tw, ta, e, pl, m->status, stream);
    case EPI_SWIGLU: return launch<EPI_SWIGLU>(tw, ta, e, pl, m->status, stream);
    case EPI_VERDICT: return launch<EPI_VERDICT>(tw, ta, e, pl, m->status, stream);
    default: return launch<EPI_QKV>(tw, ta, e, pl, m->status, stream);
  }
}

}  // namespace laser
