// Causal attention of the verify forward (Eq. 3 / Eq. 6, chain form of the mask): the K+1
// rows of a sequence against its paged bf16 KV cache, which already holds the rows' own K/V.
//
// One CTA per (sequence, head, group of TPC 16-row tiles).  A producer warp walks the sequence's
// page table and streams each 16-token page of K and V through TMA (128-byte swizzle) into a ring
// of shared-memory stages; four consumer warps compute S = Q K^T and O += P V with warp-level MMA
// (the rows are few, far below a tensor-memory tile), keep an online softmax with warp-shuffle row
// reductions, and merge their partial (max, sum, O) through shared memory at the end.  With up to
// 16 rows per sequence (TPC = 1) the four warps take pages round-robin; with more rows (K + 1 > 16
// or a large token tree, TPC = 2) two warps serve each of two row tiles and both tiles use the same
// staged page, so a page is still read from HBM once per 32 rows.  Every mbarrier wait is bounded.
//
// With few (sequence, head) pairs the walk over one sequence's pages is a latency chain that leaves most SMs idle: up to eight
// CTAs then take runs of twelve pages in turn, and the one that finishes last sums the partial results (through L2, in the order
// of the CTAs).  A cluster and distributed shared memory would merge faster, but its CTAs must find their slots together, beside
// those of the neighbouring kernels: a step of one short sequence lost 4 us a layer to that.
#include <algorithm>
#include <type_traits>

#include "mma.cuh"
#include "model.cuh"
#include "tma.cuh"

namespace laser {
namespace {

using bf16 = __nv_bfloat16;
constexpr int kConsumers = 4;
constexpr int kAttnThreads = (kConsumers + 1) * 32;
// Pages in the ring: a multiple of kConsumers, as stage s always serves warp s % 4.  A CTA's walk over its pages is paced by the bytes
// that it has in flight, so launches whose CTAs fit three an SM take the deep ring (with four, 16 sequences lose 5 % to three).
constexpr int stages_of(bool deep) { return deep ? 8 : 4; }
constexpr int kMaxPageSplits = 8;  // CTAs that share a sequence's pages
constexpr int kSplitFrom = 16;      // pages from which a split pays for the merge (about 3 us, ten pages of one CTA's walk),
constexpr int kRunPages = 12;       // and pages of a run (a multiple of kConsumers: a warp's pages stay the same ones)
constexpr int kCtasPerSm = 4;  // registers and shared memory are sized for four resident CTAs, or three with the deep ring

// SP: the pages are split over `splits` CTAs (grid x = sequences x splits).  DEEP: eight pages in the ring.  PR (precise mode): the
// queries come in fp32 (qf) and enter the score MMA as hi + lo bf16 pairs, the probabilities enter the value MMA as pairs as well,
// and the output is written as pairs ([hi | lo] rows of 2 H DH).
template <int DH, int TPC, bool PR, bool SP, bool DEEP>
__global__ void __launch_bounds__(kAttnThreads, PR && TPC == 2 && DEEP ? 2 : PR || DEEP ? 3 : kCtasPerSm)
attn_paged_kernel(const __grid_constant__ CUtensorMap kvmap, const bf16* q, const float* qf,
                  const int32_t* __restrict__ seq_ids, const int32_t* __restrict__ row_ctx,
                  const int32_t* __restrict__ row_n, int Rs, int H, int Hkv,
                  const int32_t* __restrict__ page_table, int pages_per_seq, int layer_row0,
                  bf16* __restrict__ out, int32_t* __restrict__ status,
                  const unsigned long long* row_mask, int fresh, int splits,
                  float* __restrict__ part, int32_t* __restrict__ arrived) {
  constexpr int ST = stages_of(DEEP);
  constexpr int kPartFloats = 16 * TPC * (DH + 2);   // SP: a partial result: O [rows][DH], max [rows], sum [rows]
  constexpr int HALVES = DH / 64;                 // 64-element (128-byte) column blocks per row
  constexpr int SUB = 16 * 128;                   // bytes of one 16-token x 64-element sub-tile
  constexpr int STAGE = 2 * HALVES * SUB;         // K then V
  constexpr int QLD = DH + 8;                     // padded row of the Q tile (elements)
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full_bar[ST], empty_bar[ST];
  __shared__ float s_m[kConsumers][16], s_l[kConsumers][16], s_wgt[kConsumers][16];
  __shared__ int abort_flag;
  __shared__ int s_last;
  __shared__ float s_inv[SP ? 16 * TPC : 1];

  // Programmatic dependent launch: let the next kernel start its prologue.  The kernel before this
  // one produces Q and the K/V of the step's own rows; pages that lie wholly below the committed
  // length were written by earlier steps, so the producer requests those before it waits for that
  // kernel, and the wait and the Q tile overlap their flight.  (q and qf are written while this kernel may be running already:
  // they are not const __restrict__.)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int b = SP ? blockIdx.x / splits : blockIdx.x, krank = SP ? blockIdx.x % splits : 0, h = blockIdx.y, mt = blockIdx.z;
  const int hk = h / (H / Hkv);
  const int nr = row_n[b], ctx = row_ctx[b];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int NPG = kConsumers / TPC;           // consumer warps that share a row tile (they split the pages)
  const int cta_row0 = mt * 16 * TPC;              // first row of the CTA's tiles
  const int tile = TPC == 1 ? 0 : (warp & (TPC - 1)), pgrp = TPC == 1 ? warp : (warp / TPC);
  const int row0 = cta_row0 + tile * 16;           // first row of this warp's tile
  constexpr int OW = PR ? 2 : 1;                    // output row = OW x H x DH elements
  bf16* obase = out + (size_t(b) * Rs + cta_row0) * H * DH * OW + size_t(h) * DH;
  if (cta_row0 >= nr) {  // nothing active in these tiles: zero their rows
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int idx = tid; idx < 16 * TPC * DH; idx += kAttnThreads) {
      const int r = idx / DH, d = idx % DH;
      if (cta_row0 + r < Rs) {
        obase[size_t(r) * H * DH * OW + d] = __float2bfloat16(0.f);
        if (PR) obase[size_t(r) * H * DH * OW + size_t(H) * DH + d] = __float2bfloat16(0.f);
      }
    }
    return;
  }
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles = (raw + 1023u) & ~1023u;
  uint8_t* tiles_ptr = smem_raw + (tiles - raw);
  const uint32_t q_smem = tiles + ST * STAGE;
  bf16* q_ptr = reinterpret_cast<bf16*>(tiles_ptr + ST * STAGE);
  const int n_keys = ctx + (row_mask ? nr : min(nr, cta_row0 + 16 * TPC));   // chain: no row here sees a later one
  const int all_pg = (n_keys + 15) >> 4;
  // SP: run j of the pages belongs to CTA j % splits.  Which pages a CTA sums follows from their numbers alone, neither from the
  // step's rows (a row's result is the same among drafts and alone) nor from the cache's capacity.
  const int parts = SP ? min(splits, (all_pg + kRunPages - 1) / kRunPages) : 1;
  if (SP && krank >= parts) return;
  auto page_of = [&](int p) { return SP ? ((p / kRunPages) * splits + krank) * kRunPages + p % kRunPages : p; };   // the CTA's p-th page
  auto pages_below = [&](int x) {   // how many of its pages come before page x
    if (!SP) return x;
    const int runs = x / kRunPages;
    return (runs - krank + splits - 1) / splits * kRunPages + (runs % splits == krank ? x % kRunPages : 0);
  };
  const int n_pg = pages_below(all_pg);
  const bool whole = !SP || parts == 1;
  const int unit = (b * H + h) * gridDim.z + mt;
  float* const my_part = SP ? part + size_t(unit * splits + krank) * kPartFloats : nullptr;

  if (tid == 0) {
    abort_flag = 0;
    for (int s = 0; s < ST; ++s) { mbar_init(smem_u32(&full_bar[s]), 1); mbar_init(smem_u32(&empty_bar[s]), TPC); }
    mbar_fence_init();
    tma_prefetch_map(&kvmap);
  }
  __syncthreads();   // barriers initialised

  if (warp == kConsumers) {  // producer
    if (lane == 0) {
      const int32_t* pt = page_table + size_t(seq_ids[b]) * pages_per_seq;
      // whole pages of older tokens that fit the ring (none where the kernel before may have written them)
      const int n_early = fresh ? 0 : min(pages_below(min(ctx >> 4, all_pg)), ST);
      bool ok = true;
      int issued = 0;
      const uint64_t kv_policy = make_policy_evict_first();   // a page is read once per step
      for (int p = 0; p < n_pg && ok; ++p) {
        const int s = p % ST;
        if (p == n_early) asm volatile("griddepcontrol.wait;" ::: "memory");   // from here on: pages the kernel before may write
        if (p >= ST) ok = mbar_wait(smem_u32(&empty_bar[s]), ((p / ST) - 1) & 1, &abort_flag);
        if (!ok) break;
        const uint32_t bar = smem_u32(&full_bar[s]);
        const uint32_t dst = tiles + uint32_t(s) * STAGE;
        mbar_expect_tx(bar, STAGE);
        const int phys = pt[page_of(p)];
        const int rowk = layer_row0 + ((phys * 2) * Hkv + hk) * 16;
        const int rowv = layer_row0 + ((phys * 2 + 1) * Hkv + hk) * 16;
#pragma unroll
        for (int hf = 0; hf < HALVES; ++hf) {
          tma_load_2d_hint(dst + hf * SUB, &kvmap, hf * 64, rowk, bar, kv_policy);
          tma_load_2d_hint(dst + (HALVES + hf) * SUB, &kvmap, hf * 64, rowv, bar, kv_policy);
        }
        issued = p + 1;
      }
      if (!ok)
        for (int p = max(0, issued - ST); p < issued; ++p) mbar_drain(smem_u32(&full_bar[p % ST]), (p / ST) & 1);
    }
    return;
  }

  // ---- consumers ----
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // Q tiles: rows of this sequence, zero beyond the active ones
  constexpr int QLO = 16 * TPC * QLD;             // PR: the lo parts of the Q tile follow the hi parts
  constexpr int kQLoads = 16 * TPC * (DH / 8) / (kConsumers * 32);   // (all requested before the first is used)
  uint4 qv[kQLoads][PR ? 2 : 1];
#pragma unroll
  for (int x = 0; x < kQLoads; ++x) {
    const int idx = tid + x * kConsumers * 32, r = idx / (DH / 8), c = idx % (DH / 8);
    const size_t at = (size_t(b) * Rs + cta_row0 + r) * H * DH + size_t(h) * DH + c * 8;
#pragma unroll
    for (int y = 0; y < (PR ? 2 : 1); ++y) {
      qv[x][y] = make_uint4(0, 0, 0, 0);
      if (cta_row0 + r < nr) qv[x][y] = PR ? *reinterpret_cast<const uint4*>(qf + at + 4 * y) : *reinterpret_cast<const uint4*>(q + at);
    }
  }
#pragma unroll
  for (int x = 0; x < kQLoads; ++x) {
    const int idx = tid + x * kConsumers * 32, r = idx / (DH / 8), c = idx % (DH / 8);
    uint4 v = qv[x][0];
    if (PR) {
      const float* f0 = reinterpret_cast<const float*>(&qv[x][0]);
      const float* f1 = reinterpret_cast<const float*>(&qv[x][PR ? 1 : 0]);
      const float f[8] = {f0[0], f0[1], f0[2], f0[3], f1[0], f1[1], f1[2], f1[3]};
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const __nv_bfloat162 hh = __floats2bfloat162_rn(f[2 * u], f[2 * u + 1]);
        hi[u] = *reinterpret_cast<const uint32_t*>(&hh);
        lo[u] = pack_bf16(f[2 * u] - __low2float(hh), f[2 * u + 1] - __high2float(hh));
      }
      v = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      *reinterpret_cast<uint4*>(q_ptr + QLO + r * QLD + c * 8) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
    *reinterpret_cast<uint4*>(q_ptr + r * QLD + c * 8) = v;
  }
  asm volatile("bar.sync 1, 128;" ::: "memory");
  const int g = lane >> 2, qd = lane & 3;
  const float sl2 = rsqrtf(float(DH)) * 1.4426950408889634f;
  // Q fragments are re-read from shared memory for every page: keeping them in registers
  // would cost 32 registers per thread and one resident CTA per SM
  const uint32_t q_frag = q_smem + uint32_t((tile * 16 + (lane & 7) + ((lane >> 3) & 1) * 8) * QLD + (lane >> 4) * 8) * 2;
  float o[DH / 8][4];
#pragma unroll
  for (int t = 0; t < DH / 8; ++t) o[t][0] = o[t][1] = o[t][2] = o[t][3] = 0.f;
  float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
  // last key each of this lane's two rows may see; inactive rows copy the last active row
  const int lim0 = ctx + min(row0 + g, nr - 1), lim1 = ctx + min(row0 + g + 8, nr - 1);
  // token tree: of the step's own rows a row sees those of its mask (ancestors and itself)
  const unsigned long long vis0 = row_mask ? row_mask[size_t(b) * Rs + min(row0 + g, nr - 1)] : 0ull;
  const unsigned long long vis1 = row_mask ? row_mask[size_t(b) * Rs + min(row0 + g + 8, nr - 1)] : 0ull;

  for (int p = pgrp; p < n_pg; p += NPG) {
    const int s = p % ST;
    if (!mbar_wait_warp(smem_u32(&full_bar[s]), (p / ST) & 1, &abort_flag)) break;
    const uint32_t kbase = tiles + uint32_t(s) * STAGE, vbase = kbase + HALVES * SUB;
    float sc[2][4];
#pragma unroll
    for (int t = 0; t < 2; ++t) sc[t][0] = sc[t][1] = sc[t][2] = sc[t][3] = 0.f;
    {
      const int mat = lane >> 3, key = (lane & 7) + (mat >> 1) * 8;
#pragma unroll
      for (int ks = 0; ks < DH / 16; ++ks) {
        const int c = (ks & 3) * 2 + (mat & 1);
        uint32_t kb[4], qa[4];
        ldsm_x4(qa, q_frag + ks * 32);
        ldsm_x4(kb, kbase + (ks >> 2) * SUB + key * 128 + ((c ^ (key & 7)) << 4));
        mma16816(sc[0], qa, kb[0], kb[1]);
        mma16816(sc[1], qa, kb[2], kb[3]);
        if (PR) {
          ldsm_x4(qa, q_frag + QLO * 2 + ks * 32);
          mma16816(sc[0], qa, kb[0], kb[1]);
          mma16816(sc[1], qa, kb[2], kb[3]);
        }
      }
    }
    // causal mask, online softmax (rows g and g+8 of the tile)
    const int key0 = page_of(p) * 16 + 2 * qd;
    float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int key = key0 + t * 8 + c;
        if (row_mask) {
          const int rel = key - ctx;   // >= 0: one of this step's rows (or the padding of the last page)
          if (rel >= 0 && (rel >= 64 || !((vis0 >> rel) & 1ull))) sc[t][c] = -INFINITY;
          if (rel >= 0 && (rel >= 64 || !((vis1 >> rel) & 1ull))) sc[t][2 + c] = -INFINITY;
        } else {
          if (key > lim0) sc[t][c] = -INFINITY;
          if (key > lim1) sc[t][2 + c] = -INFINITY;
        }
        mx0 = fmaxf(mx0, sc[t][c]);
        mx1 = fmaxf(mx1, sc[t][2 + c]);
      }
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1)); mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1)); mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
    const float mn0 = fmaxf(m_run[0], mx0), mn1 = fmaxf(m_run[1], mx1);
    const float mu0 = mn0 == -INFINITY ? 0.f : mn0, mu1 = mn1 == -INFINITY ? 0.f : mn1;
    const float al0 = exp2f((m_run[0] - mu0) * sl2), al1 = exp2f((m_run[1] - mu1) * sl2);
    m_run[0] = mn0; m_run[1] = mn1;
    uint32_t pf[4], pl[4] = {0u, 0u, 0u, 0u};
    float ps0 = 0.f, ps1 = 0.f;
    {
      const float p00 = exp2f((sc[0][0] - mu0) * sl2), p01 = exp2f((sc[0][1] - mu0) * sl2);
      const float p02 = exp2f((sc[0][2] - mu1) * sl2), p03 = exp2f((sc[0][3] - mu1) * sl2);
      const float p10 = exp2f((sc[1][0] - mu0) * sl2), p11 = exp2f((sc[1][1] - mu0) * sl2);
      const float p12 = exp2f((sc[1][2] - mu1) * sl2), p13 = exp2f((sc[1][3] - mu1) * sl2);
      ps0 = p00 + p01 + p10 + p11;
      ps1 = p02 + p03 + p12 + p13;
      pf[0] = pack_bf16(p00, p01);   // row g,   keys 2q..   (k low)
      pf[1] = pack_bf16(p02, p03);   // row g+8, keys 2q..
      pf[2] = pack_bf16(p10, p11);   // row g,   keys 8+2q.. (k high)
      pf[3] = pack_bf16(p12, p13);   // row g+8, keys 8+2q..
      if (PR) {
        auto lo_of = [](uint32_t packed, float a, float b) {
          const __nv_bfloat162 hh = *reinterpret_cast<const __nv_bfloat162*>(&packed);
          return pack_bf16(a - __low2float(hh), b - __high2float(hh));
        };
        pl[0] = lo_of(pf[0], p00, p01); pl[1] = lo_of(pf[1], p02, p03);
        pl[2] = lo_of(pf[2], p10, p11); pl[3] = lo_of(pf[3], p12, p13);
      }
    }
    l_run[0] = l_run[0] * al0 + ps0;
    l_run[1] = l_run[1] * al1 + ps1;
#pragma unroll
    for (int t = 0; t < DH / 8; ++t) { o[t][0] *= al0; o[t][1] *= al0; o[t][2] *= al1; o[t][3] *= al1; }
    {
      const int mat = lane >> 3, key = (lane & 7) + (mat & 1) * 8;
#pragma unroll
      for (int j = 0; j < DH / 16; ++j) {
        const int c = (j & 3) * 2 + (mat >> 1);
        uint32_t vb[4];
        ldsm_x4_t(vb, vbase + (j >> 2) * SUB + key * 128 + ((c ^ (key & 7)) << 4));
        mma16816(o[2 * j], pf, vb[0], vb[1]);
        mma16816(o[2 * j + 1], pf, vb[2], vb[3]);
        if (PR) {
          mma16816(o[2 * j], pl, vb[0], vb[1]);
          mma16816(o[2 * j + 1], pl, vb[2], vb[3]);
        }
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&empty_bar[s]));
  }

  // ---- merge the four partial results ----
  l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], 1); l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], 2);
  l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], 1); l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], 2);
  asm volatile("bar.sync 1, 128;" ::: "memory");   // every page consumed: the stages are free
  float* s_o = reinterpret_cast<float*>(tiles_ptr);  // [consumer][16][DH]
  if (qd == 0) { s_m[warp][g] = m_run[0]; s_m[warp][g + 8] = m_run[1]; s_l[warp][g] = l_run[0]; s_l[warp][g + 8] = l_run[1]; }
#pragma unroll
  for (int t = 0; t < DH / 8; ++t) {
    *reinterpret_cast<float2*>(s_o + (warp * 16 + g) * DH + t * 8 + 2 * qd) = make_float2(o[t][0], o[t][1]);
    *reinterpret_cast<float2*>(s_o + (warp * 16 + g + 8) * DH + t * 8 + 2 * qd) = make_float2(o[t][2], o[t][3]);
  }
  asm volatile("bar.sync 1, 128;" ::: "memory");
  auto store_out = [&](int rr, int d, float4 acc) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x, acc.y), hi = __floats2bfloat162_rn(acc.z, acc.w);
    *reinterpret_cast<uint2*>(obase + size_t(rr) * H * DH * OW + d) =
        make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    if (PR)   // the part of the result that the first bf16 value leaves
      *reinterpret_cast<uint2*>(obase + size_t(rr) * H * DH * OW + size_t(H) * DH + d) =
          make_uint2(pack_bf16(acc.x - __low2float(lo), acc.y - __high2float(lo)), pack_bf16(acc.z - __low2float(hi), acc.w - __high2float(hi)));
  };
  // weight of each warp's partial result per row, normalisation included: e_w / sum_w e_w l_w
  if (tid < 16 * kConsumers) {
    const int r = tid % 16, wsel = tid / 16, tsel = TPC == 1 ? 0 : (wsel & (TPC - 1));
    float mt_ = -INFINITY;
#pragma unroll
    for (int w = 0; w < kConsumers; ++w)
      if (TPC == 1 || (w & (TPC - 1)) == tsel) mt_ = fmaxf(mt_, s_m[w][r]);
    float den = 0.f, mine = 0.f;
#pragma unroll
    for (int w = 0; w < kConsumers; ++w) {
      if (TPC != 1 && (w & (TPC - 1)) != tsel) continue;
      const float e = s_m[w][r] == -INFINITY ? 0.f : exp2f((s_m[w][r] - mt_) * sl2);
      den += e * s_l[w][r];
      if (w == wsel) mine = e;
    }
    if (!whole) {      // weights against this CTA's max; the runs are weighed against each other below
      s_wgt[wsel][r] = mine;
      if (wsel == tsel) { __stcg(my_part + 16 * TPC * DH + tsel * 16 + r, mt_); __stcg(my_part + 16 * TPC * (DH + 1) + tsel * 16 + r, den); }
    } else {
      const bool live = cta_row0 + tsel * 16 + r < nr && den > 0.f && !abort_flag;
      s_wgt[wsel][r] = !live ? 0.f : SP ? mine : mine / den;
      if (SP && wsel == tsel) s_inv[tsel * 16 + r] = live ? 1.f / den : 0.f;   // (the same arithmetic as the merge of runs)
    }
  }
  asm volatile("bar.sync 1, 128;" ::: "memory");
  for (int idx = tid; idx < 16 * TPC * (DH / 4); idx += kConsumers * 32) {   // four features per thread
    const int rr = idx / (DH / 4), d = (idx % (DH / 4)) * 4;      // rr: row within the CTA's tiles
    const int tsel = rr / 16, r = rr % 16;
    if (cta_row0 + rr >= Rs) continue;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < kConsumers; ++w) {
      if (TPC != 1 && (w & (TPC - 1)) != tsel) continue;
      const float e = s_wgt[w][r];
      const float4 x = *reinterpret_cast<const float4*>(s_o + (w * 16 + r) * DH + d);
      acc.x += e * x.x; acc.y += e * x.y; acc.z += e * x.z; acc.w += e * x.w;
    }
    if (SP && whole) { const float inv = s_inv[rr]; acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv; }
    if (whole) store_out(rr, d, acc);
    else __stcg(reinterpret_cast<float4*>(my_part + rr * DH + d), acc);
  }
  if (!whole) {
    asm volatile("bar.sync 1, 128;" ::: "memory");
    if (tid == 0) {
      __threadfence();
      s_last = atomicAdd(arrived + unit, 1) == parts - 1;
      __threadfence();
      if (s_last) arrived[unit] = 0;      // for the next layer
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    if (s_last) {   // a warp a row, four features a lane
      const float* first = part + size_t(unit * splits) * kPartFloats;
      for (int rr = warp; rr < 16 * TPC && cta_row0 + rr < Rs; rr += kConsumers) {
        float mx[kMaxPageSplits], den[kMaxPageSplits];
        float4 x[kMaxPageSplits];
#pragma unroll
        for (int q = 0; q < kMaxPageSplits; ++q) {
          const float* pq = first + size_t(min(q, parts - 1)) * kPartFloats;
          mx[q] = __ldcg(pq + 16 * TPC * DH + rr);
          den[q] = __ldcg(pq + 16 * TPC * (DH + 1) + rr);
          x[q] = 4 * lane < DH ? __ldcg(reinterpret_cast<const float4*>(pq + rr * DH + 4 * lane)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        float top = -INFINITY, total = 0.f;
#pragma unroll
        for (int q = 0; q < kMaxPageSplits; ++q) if (q < parts) top = fmaxf(top, mx[q]);
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < kMaxPageSplits; ++q) {
          const float e = q < parts && mx[q] > -INFINITY ? exp2f((mx[q] - top) * sl2) : 0.f;
          total += e * den[q];
          acc.x += e * x[q].x; acc.y += e * x[q].y; acc.z += e * x[q].z; acc.w += e * x[q].w;
        }
        const float inv = cta_row0 + rr < nr && total > 0.f && !abort_flag ? 1.f / total : 0.f;
        acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
        if (4 * lane < DH) store_out(rr, 4 * lane, acc);
      }
    }
  }
  if (tid == 0 && abort_flag) atomicCAS(status, 0, LASER_ERR_TIMEOUT);
}

}  // namespace

bool attention_tma_supported(const laser_model* m, const laser_kv* kv) {
  return kv->has_pages_map && (m->cfg.head_dim == 64 || m->cfg.head_dim == 128);
}

laser_status attention_tma_launch(laser_model* m, laser_kv* kv, int layer, const int32_t* seq_ids, int B, int Rs, bool tree, bool fresh,
                                  cudaStream_t stream) {
  const int dh = m->cfg.head_dim, H = m->cfg.n_heads, Hkv = m->cfg.n_kv_heads;
  const int64_t rows_per_layer = int64_t(kv->n_pages) * 2 * Hkv * 16;
  const int layer_row0 = int(rows_per_layer * layer);
  const int tiles = ceil_div(Rs, 16), tpc = tiles > 1 ? 2 : 1;   // row tiles of a sequence; tiles per CTA
  // Page splits while the CTAs stay resident, where the cache can hold pages enough; what a sequence has is known on the device
  // alone, and CTAs that find no run to take leave.  7B, 6 layers, steps of 9 rows, 128 / 256 / 512 / 1000 cached tokens in a cache of 256
  // pages a sequence, us; unsplit with a ring of four: one sequence 526 / 544 / 580 / 649, two 551 / 569 / 606 / 679, four 612 / 630 / 665 /
  // 734, eight 645 / 664 / 703 / 787; here, in eight 516 / 540 / 545 / 553, in six 539 / 569 / 576 / 581, in three 605 / 635 / 648 / 675, unsplit
  // with the deep ring 640 / 656 / 680 / 736.  A ring of four and runs of eight pages: one sequence 543 / 545 / 551 / 563, four 635 / 643 /
  // 659 / 687: the merge costs 3 us a layer, which a text of two runs does not win back.  Runs of 8 or 16 pages with the deep ring: one
  // sequence 535 / 539 / 546 / 553, 518 / 551 / 557 / 565.  Caches that hold less than 32 pages are split for up to 74 pairs of sequence
  // and head (256 tokens in such a cache: two sequences 584 unsplit, 575 in six; four 623 unsplit, 644 in three).  (A prefill's
  // chunks are many.)
  const bool pr = m->precise;
  const int units = B * H * ceil_div(tiles, tpc), most = kv->pages_per_seq;
  const int resident = pr && tpc == 2 ? kAttnSplitCtas / 3 * 2 : kAttnSplitCtas;   // (hi + lo queries of 32 rows take more shared memory)
  const bool deep = !fresh && units <= resident;
  const int splits = !deep || most < (units <= kAttnSplitCtas / 6 ? kSplitFrom : 2 * kSplitFrom) ? 1 : std::min(kMaxPageSplits, resident / units);
  const size_t smem = 1024 + size_t(stages_of(deep)) * (2 * (dh / 64) * 16 * 128) + size_t(16) * tpc * (dh + 8) * 2 * (pr ? 2 : 1);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(B * splits), unsigned(H), unsigned(ceil_div(tiles, tpc)));
  cfg.blockDim = dim3(kAttnThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const __nv_bfloat16* q = m->q;
  const int32_t *rc = m->row_ctx, *rn = m->row_n, *pt = kv->page_table;
  const unsigned long long* mask = tree ? m->row_mask : nullptr;
  const float* qf = m->qf;
  auto launch = [&](auto kernel) -> laser_status {
    LASER_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
    LASER_CUDA(cudaLaunchKernelEx(&cfg, kernel, kv->pages_map, q, qf, seq_ids, rc, rn, Rs, H, Hkv, pt, kv->pages_per_seq, layer_row0,
                                  m->attn, m->status, mask, fresh ? 1 : 0, splits, m->attn_part, m->attn_arrived));
    return LASER_OK;
  };
  auto by_split = [&](auto dh_tag, auto tpc_tag, auto pr_tag) -> laser_status {
    constexpr int D = decltype(dh_tag)::value, T = decltype(tpc_tag)::value;
    constexpr bool P = decltype(pr_tag)::value;
    return splits > 1 ? launch(attn_paged_kernel<D, T, P, true, true>) : deep ? launch(attn_paged_kernel<D, T, P, false, true>) : launch(attn_paged_kernel<D, T, P, false, false>);
  };
  auto by_mode = [&](auto dh_tag, auto tpc_tag) { return pr ? by_split(dh_tag, tpc_tag, std::true_type{}) : by_split(dh_tag, tpc_tag, std::false_type{}); };
  using std::integral_constant;
  auto by_rows = [&](auto dh_tag) { return tpc == 1 ? by_mode(dh_tag, integral_constant<int, 1>{}) : by_mode(dh_tag, integral_constant<int, 2>{}); };
  LASER_TRY(dh == 128 ? by_rows(integral_constant<int, 128>{}) : by_rows(integral_constant<int, 64>{}));
  count_launch();
  LASER_CUDA(cudaGetLastError());
  return LASER_OK;
}

}  // namespace laser
