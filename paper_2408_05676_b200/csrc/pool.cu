// Customized Retrieval Pool (Section 3.2) and draft retrieval, Retrieve(D, tail, K) of Eq. 5
// (Section 3.3).
//
// Index: for every n in [n_min, n_max] an open-addressing hash table keyed by a 64-bit hash of
// (group, n-gram) whose 8-byte entries {low half of the key, start} point at a run of a position
// array; the last position of a run carries a mark.  A run lists, ascending, every position where
// that n-gram ends inside that group - exactly the nodes a per-group trie reaches with the n-gram as
// prefix, with multiplicity.  Every group has a region of the table for itself (region_of), so that
// a group is indexed on its own, and a key's home slot is its high half scaled to the region.
// Equal halves of different keys only cost a look at the wrong run, a collision of whole keys only
// merges runs: every position read at lookup time is checked against the actual pool tokens and the
// group bounds, so results never depend on the hash.
//
// Build: a group whose working set fits shared memory is indexed there by one CTA per n
// (index_group_kernel); the n-grams of larger groups, and of many tiny ones, are inserted into the table itself, and their
// positions sorted by slot, all groups together, with the radix sort of CUB, the header library
// shipped with the CUDA toolkit (nothing on the per-step path uses it).
//
// Lookup: one warp per query.  Four suffix lengths are probed at once; where that does not settle one, all 32 lanes probe 32
// consecutive slots (256 B, coalesced); the run is read 32 positions at a time, verified, and compacted; the greedy
// highest-frequency walk votes over at most 64 occurrences held two per lane.  Queries that
// need more than 64 occurrences (max_occ = 0 or > 64) go to a work list served by teams of 256 threads and by whole CTAs.
#include <cub/device/device_radix_sort.cuh>

#include <algorithm>
#include <memory>
#include <new>
#include <type_traits>

#include "common.cuh"

struct laser_pool {
  int64_t n_tokens = 0;
  int32_t n_groups = 0, n_min = 0, n_max = 0;
  int32_t vocab_bound = 0;  // largest token id + 1
  int device = 0;
  void* memory = nullptr;            // the one device allocation that holds all of the below
  int32_t* tokens = nullptr;         // dev [n_tokens]
  int64_t* group_offsets = nullptr;  // dev [n_groups + 1]
  struct Level {
    uint2* table = nullptr;          // {key's low half, start of its run}, all ones = empty
    uint32_t* positions = nullptr;   // [n_tokens + 32], runs end with a marked position
    int64_t n_keys = 0;
  } level[9];                        // indexed by n
  int64_t device_bytes = 0;
};

namespace laser {
namespace {

constexpr int kMaxN = 8;
constexpr int kMaxK = 64;
constexpr uint64_t kEmpty = ~0ULL;
constexpr uint32_t kRunEnd = 0x80000000u;   // mark of a run's last position (positions are below 2^31)

// Two 32-bit hashes side by side, each a polynomial in the tokens that is mixed once (the finalizer of MurmurHash3): a 64-bit one took
// two and a half times the multiplications, and hashing was an eighth of the build in shared memory.  The upper gives a key's
// home slot, the lower is what its entry shows of it.
__host__ __device__ __forceinline__ uint32_t mix32(uint32_t x) {
  x ^= x >> 16; x *= 0x85ebca6bu;
  x ^= x >> 13; x *= 0xc2b2ae35u;
  return x ^ (x >> 16);
}
__host__ __device__ __forceinline__ uint64_t key_of(uint32_t hi, uint32_t lo) { return uint64_t(hi) << 32 | lo; }
__host__ __device__ __forceinline__ uint64_t key_begin(int g, int n) { return key_of(uint32_t(g) * 8u + uint32_t(n), uint32_t(g)); }
__host__ __device__ __forceinline__ uint64_t key_push(uint64_t h, int32_t tok) {
  return key_of(uint32_t(h >> 32) * 0x9E3779B1u + uint32_t(tok), uint32_t(h) * 0x85EBCA77u + uint32_t(tok));
}
__host__ __device__ __forceinline__ uint64_t key_end(uint64_t h) { return key_of(mix32(uint32_t(h >> 32)), mix32(uint32_t(h))); }
__device__ __forceinline__ uint32_t home_slot(uint64_t key, uint32_t slots) { return __umulhi(uint32_t(key >> 32), slots); }

// A group's region of a table: 13 slots per 8 tokens, and always one more than there are tokens.
struct Region { int64_t base; uint32_t slots; };
__host__ __device__ __forceinline__ int64_t region_base(int64_t group_start, int64_t g) { return group_start + (group_start >> 1) + (group_start >> 3) + 2 * g; }
__host__ __device__ __forceinline__ Region region_of(int64_t lo, int64_t hi, int g) {
  const int64_t base = region_base(lo, g);
  return Region{base, uint32_t(region_base(hi, int64_t(g) + 1) - base)};
}

constexpr int kKeyThreads = 256;

struct IndexLevels { uint2* table[kMaxN + 1]; uint32_t* positions[kMaxN + 1]; };

// The groups that the sort takes: their ids, and where the positions of each begin when they are laid end to end.
// (null lists: all groups are, in their own order)
struct SortedGroups {
  const uint32_t *id, *at;
  int n;
  __device__ __forceinline__ int group(int l) const { return id ? int(id[l]) : l; }
  __device__ __forceinline__ int64_t start(const int64_t* __restrict__ goff, int l) const { return at ? int64_t(at[l]) : goff[l]; }
};

// Largest l in [lo, hi) with start(l) <= i (skips empty groups)
__device__ __forceinline__ int group_of(const SortedGroups& lg, const int64_t* __restrict__ goff, int lo, int hi, int64_t i) {
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (lg.start(goff, mid) <= i) lo = mid; else hi = mid;
  }
  return lo;
}

// Inserts the n-grams of the listed groups, for the n from n0 on, into their regions (cleared before) and leaves every (n,
// position) with the number of its n-gram's slot among all those tables' (kNoSlot where none ends).  An entry is {key's low
// half, a position of the n-gram} here; equal low halves are told apart by the tokens.  A block's positions are consecutive: two
// searches bound the groups of its threads, and as they are a chain of loads a block takes kInsertItems positions a thread (2.8 M
// positions, four n: 374 us with one, 256 with four).  Bound by the latency of the probes, in L2 for the most part.
constexpr uint32_t kNoSlot = 0xffffffffu;
constexpr int kInsertItems = 4, kInsertBlock = kInsertItems * kKeyThreads;
__global__ void __launch_bounds__(kKeyThreads)
insert_sorted_kernel(const int32_t* __restrict__ tok, const int64_t* __restrict__ goff, SortedGroups lg, int64_t M, int n0,
                    const IndexLevels lv, uint32_t table_slots, uint32_t* __restrict__ slot_of, uint32_t* __restrict__ pos,
                    unsigned long long* __restrict__ n_valid, int* __restrict__ max_tok) {
  __shared__ int s_g[2], s_max[kKeyThreads / 32];
  __shared__ unsigned s_ends;
  const int64_t i0 = int64_t(blockIdx.x) * kInsertBlock;
  const int n = n0 + blockIdx.y;
  unsigned long long* const table = reinterpret_cast<unsigned long long*>(lv.table[n]);
  if (threadIdx.x < 2) s_g[threadIdx.x] = group_of(lg, goff, 0, lg.n, min(M - 1, i0 + threadIdx.x * (kInsertBlock - 1)));
  if (threadIdx.x == 0) s_ends = 0;
  __syncthreads();
  int mt = -1, ends = 0;
  for (int64_t i = i0 + threadIdx.x; i < min(M, i0 + kInsertBlock); i += kKeyThreads) {
    const int l = s_g[0] == s_g[1] ? s_g[0] : group_of(lg, goff, s_g[0], s_g[1] + 1, i), g = lg.group(l);
    const int64_t lo = goff[g], inside = i - lg.start(goff, l), p = lo + inside;
    bool valid = inside >= n - 1;
    uint64_t key = key_begin(g, n);
    if (valid)
      for (int j = 0; j < n; ++j) {
        const int32_t t = tok[p - n + 1 + j];
        if (t < 0) { valid = false; break; }
        key = key_push(key, t);
      }
    uint32_t at = kNoSlot;
    if (valid) {
      key = key_end(key);
      const Region rg = region_of(lo, goff[g + 1], g);
      const unsigned long long entry = (uint64_t(uint32_t(p)) << 32) | uint32_t(key);
      uint32_t s = home_slot(key, rg.slots);
      for (uint32_t tries = 0; tries < rg.slots; ++tries) {   // there are more slots than positions
        unsigned long long* e = table + rg.base + s;
        unsigned long long old = __ldcg(e);
        if (old == kEmpty) {
          old = atomicCAS(e, (unsigned long long)kEmpty, entry);
          if (old == kEmpty) break;
        }
        if (uint32_t(old) == uint32_t(key)) {
          const int64_t q = int64_t(old >> 32);
          bool same = true;
          for (int j = 0; same && j < n; ++j) same = tok[p - j] == tok[q - j];
          if (same) break;
        }
        if (++s == rg.slots) s = 0;
      }
      at = blockIdx.y * table_slots + uint32_t(rg.base) + s;
      ++ends;
    }
    slot_of[blockIdx.y * M + i] = at;
    pos[blockIdx.y * M + i] = uint32_t(p);
    mt = max(mt, tok[p]);
  }
  ends = __reduce_add_sync(0xffffffffu, ends);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_ends, unsigned(ends));
  __syncthreads();
  if (threadIdx.x == 0 && s_ends) atomicAdd(n_valid + n, (unsigned long long)s_ends);
  if (blockIdx.y == 0) {
    for (int o = 16; o; o >>= 1) mt = max(mt, __shfl_xor_sync(0xffffffffu, mt, o));
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = mt;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < kKeyThreads / 32; ++w) mt = max(mt, s_max[w]);
      if (mt > *max_tok) atomicMax(max_tok, mt);
    }
  }
}

// (slot, position) pairs sorted by slot to the position arrays (from `first` on) with their run marks, and the start of every
// run to its slot.
__global__ void __launch_bounds__(kKeyThreads)
index_runs_kernel(const uint32_t* __restrict__ slot, const uint32_t* __restrict__ pos, int64_t count, int64_t first, int n0,
                  const IndexLevels lv, uint32_t table_slots, const unsigned long long* __restrict__ n_valid,
                  unsigned long long* __restrict__ n_heads) {
  __shared__ unsigned s_heads[kMaxN + 1];
  if (threadIdx.x <= kMaxN) s_heads[threadIdx.x] = 0;
  __syncthreads();
  const int64_t i = int64_t(blockIdx.x) * kKeyThreads + threadIdx.x;
  const uint32_t s = i < count ? slot[i] : kNoSlot;
  if (s != kNoSlot) {
    const uint32_t l = s / table_slots;
    int64_t rank = i;                      // among the positions of its n
    for (uint32_t x = 0; x < l; ++x) rank -= int64_t(n_valid[n0 + x]);
    const bool end = i + 1 == count || slot[i + 1] != s;
    lv.positions[n0 + l][first + rank] = pos[i] | (end ? kRunEnd : 0u);
    if (i == 0 || slot[i - 1] != s) {
      lv.table[n0 + l][s - l * table_slots].y = uint32_t(first + rank);
      atomicAdd(&s_heads[n0 + l], 1u);
    }
  }
  __syncthreads();
  if (threadIdx.x <= kMaxN && s_heads[threadIdx.x]) atomicAdd(n_heads + threadIdx.x, (unsigned long long)s_heads[threadIdx.x]);
}

__global__ void __launch_bounds__(kKeyThreads)
clear_regions_kernel(const IndexLevels lv, int n_min, const int64_t* __restrict__ goff, SortedGroups lg, int first) {
  const int g = lg.group(first + blockIdx.y);
  const Region rg = region_of(goff[g], goff[g + 1], g);
  uint2* table = lv.table[n_min + blockIdx.z] + rg.base;
  for (uint32_t s = blockIdx.x * kKeyThreads + threadIdx.x; s < rg.slots; s += gridDim.x * kKeyThreads) table[s] = make_uint2(0xffffffffu, 0xffffffffu);
}

// ---- a group in shared memory ------------------------------------------------------------
// One CTA per (group, n): the region's slots as words, into which the group's n-grams are inserted (told apart by 16 bits of their
// key, then by their tokens); the counts of the slots become run starts by a prefix sum; a block of positions after the other
// goes into the runs, and a position finds its place among those of its block by counting.  Memory sees the tokens, the runs and
// the regions; what bounds the kernel is the latency of its steps in shared memory.  In the insert loop a lane takes the warp's
// next position as soon as it has placed one: with positions of its own for every lane the CTA waits for the unluckiest of 512
// probe walks, and with a warp in step for the longest of 32, four times as long again.
// Groups come in three classes by size, for one, two and three CTAs an SM.  10 M tokens in 2000 groups, four levels: 690 us for
// the 72 % of them in groups that fit (805 with positions per lane, representatives' tokens compared at every probe and a 64-bit
// hash) and 735 us for the rest, against 4.7 ms for a sort of all positions by 64-bit key and n; the whole build 4.99 -> 1.49 ms.
constexpr uint32_t kFreeWord = 0xffffffffu;
constexpr int kScan = 128;                       // slots that a warp scans at a time
constexpr size_t group_smem(int64_t tokens) {    // words, tokens, slot and run member of every position
  return size_t((tokens + tokens / 2 + tokens / 8 + 4 + kScan - 1) / kScan * kScan) * 4 + size_t(tokens) * 8 + 16;
}
constexpr int kClasses = 3;
constexpr int kGroupMax = 15400;                 // tokens of the largest group
constexpr int64_t kClassMax[kClasses] = {kGroupMax, 7600, 4900};
static_assert(group_smem(kGroupMax) <= 226 * 1024 && 2 * group_smem(kClassMax[1]) <= 224 * 1024 && 3 * group_smem(kClassMax[2]) <= 222 * 1024 &&
              kGroupMax + kGroupMax / 2 + kGroupMax / 8 + 4 < 65535, "");

// A CTA per (group, n) costs about 15 ns of the device whatever the group's size, so tiny groups are sorted with the large ones
// where they are so many that the sort's own launches (0.2 ms) do not show.  10 M tokens in groups of 2 / 5 / 10 / 100 / 200 / 250: a
// CTA each 255 / 92 / 48 / 6.9 / 3.95 / 3.31 ms, sorted 11 / 5.4 / 4.0 / 3.1 / 3.24 / 3.13; 1 M tokens in groups of 10 / 100 / 200: 4.4 / 0.71 /
// 0.46, sorted 0.53 / 0.45 / 0.46; 200 k tokens in groups of 20 / 100 (2000 of them): 0.54 / 0.21, sorted 0.25 / 0.21.
constexpr int kTinyGroup = 256, kManyTiny = 4096;

template <int THREADS, int CTAS>
__global__ void __launch_bounds__(THREADS, CTAS)
index_group_kernel(const int32_t* tok, const int64_t* goff, const uint32_t* group_id, const uint32_t* group_at, int leads, int n_min,
                   const IndexLevels lv, unsigned long long* n_heads, int* max_tok) {
  constexpr int kWarps = THREADS / 32;
  extern __shared__ __align__(16) uint32_t s_word[];
  __shared__ uint32_t s_sum[kWarps];
  __shared__ int s_heads;
  if (leads) wait_for_earlier();  // the first class waits for its inputs, and so do those that it lets start
  next_may_launch();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = int(group_id[blockIdx.x]), n = n_min + blockIdx.y;
  const int64_t lo = goff[g], hi = goff[g + 1], first = group_at[blockIdx.x];   // first: of the group's runs
  const int T = int(hi - lo);
  const Region rg = region_of(lo, hi, g);
  const int slots = int(rg.slots), words = (slots + kScan - 1) / kScan * kScan;
  int32_t* s_tok = reinterpret_cast<int32_t*>(s_word + words);
  uint16_t* s_slot = reinterpret_cast<uint16_t*>(s_tok + T);
  uint16_t* s_member = s_slot + T;
  uint2* const table = lv.table[n] + rg.base;

  if (tid == 0) s_heads = 0;
  for (int s = tid; s < words; s += THREADS) s_word[s] = kFreeWord;
  for (int s = tid; s < slots; s += THREADS) table[s] = make_uint2(0xffffffffu, 0xffffffffu);
  int mt = -1;
  for (int i = tid; i < T; i += THREADS) {
    const int32_t t = tok[lo + i];
    s_tok[i] = t;
    mt = max(mt, t);
  }
  if (blockIdx.y == 0) {
    for (int o = 16; o; o >>= 1) mt = max(mt, __shfl_xor_sync(0xffffffffu, mt, o));
    if (lane == 0 && mt > *max_tok) atomicMax(max_tok, mt);
  }
  __syncthreads();
  auto ngram_key = [&](int i) {      // of the n-gram that ends at i
    uint64_t h = key_begin(g, n);
    for (int j = i - n + 1; j <= i; ++j) h = key_push(h, s_tok[j]);
    return key_end(h);
  };

  // home slots, and 16 bits of the keys where the runs' members will be
  for (int i = tid; i < T; i += THREADS) {
    uint64_t h = key_begin(g, n);
    int32_t least = i >= n - 1 ? 0 : -1;
    for (int j = max(i - n + 1, 0); j <= i; ++j) {
      const int32_t t = s_tok[j];
      least = min(least, t);
      h = key_push(h, t);
    }
    h = key_end(h);
    s_slot[i] = least >= 0 ? uint16_t(home_slot(h, rg.slots)) : uint16_t(0xffff);
    s_member[i] = uint16_t(h);
  }
  // insert: words of {16 bits of the key | position}, so that another n-gram's slot is passed without a look at its tokens.  A
  // warp's positions are those that its threads hashed; its lanes take them as they become free, for some walks are long
  // (with twelve positions to each lane the CTA waited for the unluckiest of its 512).
  __syncwarp();
  {
    auto position = [&](int j) { return (j >> 5) * THREADS + warp * 32 + (j & 31); };
    int i = position(lane), given = 32;
    int s = i < T ? s_slot[i] : 0;
    while (__any_sync(0xffffffffu, i < T)) {
      bool placed = i < T && s == 0xffff;       // (none ends here)
      if (i < T && !placed) {                   // (there are more slots than positions)
        const uint32_t word = uint32_t(s_member[i]) << 16 | uint32_t(i);
        uint32_t w = *const_cast<volatile uint32_t*>(s_word + s);
        if (w == kFreeWord) {
          w = atomicCAS(s_word + s, kFreeWord, word);
          placed = w == kFreeWord;
        }
        if (!placed && (w ^ word) < 0x10000u) {
          const int rep = int(w & 0xffffu);
          placed = true;
          for (int j = 0; j < n; ++j) placed = placed && s_tok[i - j] == s_tok[rep - j];
        }
      }
      const unsigned done = __ballot_sync(0xffffffffu, placed);
      if (placed) {
        s_slot[i] = uint16_t(s);
        i = position(given + __popc(done & ((1u << lane) - 1)));
        if (i < T) s = s_slot[i];
      } else if (++s == slots) {
        s = 0;
      }
      given += __popc(done);
    }
  }
  __syncthreads();
  for (int s = 4 * tid; s < words; s += 4 * THREADS) *reinterpret_cast<uint4*>(s_word + s) = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  for (int i = tid; i < T; i += THREADS)
    if (s_slot[i] != 0xffff) atomicAdd(s_word + s_slot[i], 0x10000u);
  __syncthreads();

  // counts -> {0 | start}: a warp's share of the slots is consecutive, four a lane at a time
  const int per = (words / kScan + kWarps - 1) / kWarps * kScan, s0 = min(words, warp * per), s1 = min(words, s0 + per);
  uint32_t sum = 0, heads = 0;
  for (int s = s0 + lane; s < s1; s += 32) {
    const uint32_t c = s_word[s] >> 16;
    sum += c;
    heads += c != 0;
  }
  sum = __reduce_add_sync(0xffffffffu, sum);
  heads = __reduce_add_sync(0xffffffffu, heads);
  if (lane == 0) { s_sum[warp] = sum; if (heads) atomicAdd(&s_heads, int(heads)); }
  __syncthreads();
  uint32_t start = 0, total = 0;
  for (int w = 0; w < kWarps; ++w) { if (w < warp) start += s_sum[w]; total += s_sum[w]; }
  for (int s = s0; s < s1; s += kScan) {
    uint4* at = reinterpret_cast<uint4*>(s_word + s) + lane;
    const uint4 w = *at;
    const uint32_t c0 = w.x >> 16, c1 = c0 + (w.y >> 16), c2 = c1 + (w.z >> 16), c3 = c2 + (w.w >> 16);
    uint32_t upto = c3;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, upto, o);
      if (lane >= o) upto += v;
    }
    const uint32_t at0 = start + upto - c3;
    *at = make_uint4(at0, at0 + c0, at0 + c1, at0 + c2);
    start += __shfl_sync(0xffffffffu, upto, 31);
  }
  __syncthreads();

  // every position into its run: blocks of 128 or 256 positions in order, within a block in the order of arrival; the words
  // become {count | start}.  (A large block is placed quickly, a small one ranked: groups of 4,900 to 7,600 tokens, n = 1,
  // blocks of 512 take 4 and 62 thousand cycles, of 256 7 and 41, of 128 12 and 28, of 32 by a warp alone 38 and 17; n = 4, 4 and 13, 6
  // and 13, 11 and 13, 39 and 13.)
  const uint32_t block_bits = n == 1 ? 7 : 8, in_block = 1u << block_bits;
  if (uint32_t(tid) < in_block)
    for (int i0 = 0; i0 < T; i0 += int(in_block)) {
      const int i = i0 + tid, s = i < T ? s_slot[i] : 0xffff;
      if (s != 0xffff) {
        const uint32_t w = atomicAdd(s_word + s, 0x10000u);
        s_member[(w & 0xffffu) + (w >> 16)] = uint16_t(i);
      }
      asm volatile("bar.sync 1, %0;" ::"r"(in_block) : "memory");
    }
  __syncthreads();

  // to its place in the run, behind those of earlier blocks; the first of a run makes its entry
  uint32_t* positions = lv.positions[n] + first;
  for (uint32_t k = tid; k < total; k += THREADS) {
    const uint32_t i = s_member[k], block = i >> block_bits, s = s_slot[i], w = s_word[s], begin = w & 0xffffu, end = begin + (w >> 16);
    uint32_t left = k, smaller = 0;
    while (left > begin) {
      const uint32_t m = s_member[left - 1];
      if (m >> block_bits != block) break;
      smaller += m < i;
      --left;
    }
    for (uint32_t r = k + 1; r < end; ++r) {
      const uint32_t m = s_member[r];
      if (m >> block_bits != block) break;
      smaller += m < i;
    }
    const uint32_t at = left + smaller;
    positions[at] = (uint32_t(lo) + i) | (at + 1 == end ? kRunEnd : 0u);
    if (k == begin) table[s] = make_uint2(uint32_t(ngram_key(int(i))), uint32_t(first) + begin);
  }
  if (tid == 0 && s_heads) atomicAdd(n_heads + n, (unsigned long long)s_heads);
  wait_for_earlier();             // (the classes are independent; what follows in the stream waits for all)
}

// ---------------------------------------------------------------------------------------
struct PoolView {
  const int32_t* tok;
  const int64_t* goff;
  int G;
  const uint2* table[kMaxN + 1];
  const uint32_t* positions[kMaxN + 1];
};

PoolView view_of(const laser_pool* pool) {
  PoolView pv{};
  pv.tok = pool->tokens; pv.goff = pool->group_offsets; pv.G = pool->n_groups;
  for (int n = pool->n_min; n <= pool->n_max; ++n) {
    pv.table[n] = pool->level[n].table;
    pv.positions[n] = pool->level[n].positions;
  }
  return pv;
}

struct DraftArgs {
  const int32_t* tails; const int32_t* tail_len; const int32_t* group_id;
  int B, K, n_min, n_max, min_draft, max_occ;
  int32_t* draft; int32_t* draft_len; int32_t* match_n;
  int32_t* work;       // large-run path: WORK_HEAD counters (zero between calls), then the items
  int64_t n_positions;
};

// Warp-cooperative probe: the next slot, `off` or more past the key's home, whose entry carries the key's low half.  Returns
// false when an empty slot comes first (linear probing without deletions: the key is not behind it); else `off` is that slot's.
__device__ __forceinline__ bool probe(const uint2* __restrict__ table, uint32_t slots, uint64_t key, int lane, uint32_t& off,
                                      uint32_t& start) {
  const uint32_t home = home_slot(key, slots);
  for (; off < slots; off += 32) {
    uint64_t s = uint64_t(home) + off + lane;   // (a small region is seen more than once: up to its first empty slot, it counts)
    if (s >= slots) s %= slots;
    const uint2 e = __ldg(&table[s]);
    const unsigned empty = __ballot_sync(0xffffffffu, e.x == 0xffffffffu && e.y == 0xffffffffu);
    unsigned hit = __ballot_sync(0xffffffffu, e.x == uint32_t(key) && e.y != 0xffffffffu);
    if (empty) hit &= (empty & -empty) - 1u;
    if (hit) {
      const int src = __ffs(hit) - 1;
      start = __shfl_sync(0xffffffffu, e.y, src);
      off += src;
      return true;
    }
    if (empty) return false;
  }
  return false;
}

__device__ __forceinline__ bool is_occurrence(const int32_t* __restrict__ tok, int64_t lo, int64_t hi,
                                              int64_t p, const int32_t* tail, int n) {
  if (p - n + 1 < lo || p >= hi) return false;
  for (int j = 0; j < n; ++j)
    if (tok[p - n + 1 + j] != tail[j]) return false;
  return true;
}

// The same, and the token at p + j (-1 beyond the group; p >= lo): up to four of the tail's are asked for together with it, for they are
// mostly of one sector of memory, which with most of an SM's shared memory in use is gone again when it is asked for a second time.
__device__ __forceinline__ bool occurrence_and_next(const int32_t* __restrict__ tok, int64_t lo, int64_t hi, int64_t p, const int32_t* tail,
                                                    int n, int j, int32_t& next) {
  constexpr int kAtOnce = 4;
  const bool in = p - n + 1 >= lo && p < hi;
  int32_t w[kAtOnce];
#pragma unroll
  for (int x = 0; x < kAtOnce; ++x) w[x] = in && x < n ? tok[p - x] : 0;
  next = in && p + j < hi ? tok[p + j] : -1;
  bool ok = in;
#pragma unroll
  for (int x = 0; x < kAtOnce; ++x) ok = ok && (x >= n || w[x] == tail[n - 1 - x]);
  for (int x = kAtOnce; ok && x < n; ++x) ok = tok[p - x] == tail[n - 1 - x];
  return ok;
}

// The group's occurrences of the n tail tokens, ascending, behind the n_occ that s_occ[64] already holds, until there are
// `cap` (more may be counted, 64 are kept).  All lanes of a warp.  start: of their run, if there is one.  off: slots past the home one
// that are known not to be the key's.
__device__ __forceinline__ int gather_occurrences(const PoolView& pv, int64_t lo, int64_t hi, const int32_t* tail, int n, uint64_t key,
                                                  int g, int lane, uint32_t* s_occ, int n_occ, int cap, uint32_t& start, uint32_t off = 0) {
  const int before = n_occ;
  const Region rg = region_of(lo, hi, g);
  for (; n_occ < cap && n_occ == before && probe(pv.table[n] + rg.base, rg.slots, key, lane, off, start); ++off) {
    for (uint32_t base = start; n_occ < cap; base += 32) {   // (the array is padded: lanes past its end read marked padding)
      const uint32_t v = pv.positions[n][base + lane];
      const unsigned ends = __ballot_sync(0xffffffffu, (v & kRunEnd) != 0);
      const int64_t p = int64_t(v & ~kRunEnd);
      const bool ok = (!ends || lane < __ffs(ends)) && is_occurrence(pv.tok, lo, hi, p, tail, n);
      const unsigned ball = __ballot_sync(0xffffffffu, ok);
      const int slot = n_occ + __popc(ball & ((1u << lane) - 1));
      if (ok && slot < 64) s_occ[slot] = uint32_t(p);
      n_occ += __popc(ball);
      if (ends) break;
    }
  }
  return n_occ;
}

// The greedy highest-frequency walk over up to 64 occurrences, two a lane (e0, e1; alive a0, a1), from depth `len` on (their
// tokens up to there agree): at every depth the most frequent next token, ties to the smallest, and the occurrences that
// continue with it.  An occurrence is a pool position, or with bit 31 an index into the history h[0 .. hl).  Writes the
// tokens to s_cur and returns the depth reached, at most K.  s_val: kWalkVals words, 16-byte aligned.  All lanes of a warp.
// Up to four occurrences are read along: a lane a depth, 32 of them held in registers, so that one step covers all depths where they agree, and
// a vote follows where they part.  More of them vote a depth at a time on tokens of which eight depths are requested together: first
// for the token of the first of them, which a majority ends, then each lane compares its tokens with all of them.
// Bound by latency and by the fetch of the code, which most warps go through once.  4096 queries on 50 M tokens, max_occ 64, a batch asked
// again: 15.1 us with votes whose steps are the distinct tokens, one depth after the other; 12.6 with eight occurrences read along,
// loaded again wherever they part, no look for a majority and four depths requested; 11.5 as it is (10.9 with eight held in registers).
// Where many occurrences agree for long - 512 queries on groups of 200 thousand tokens - 13.6, 18.3 and 14.4 us (16.2 with eight held).
constexpr int kWalkFew = 4, kWalkDepths = 8, kWalkVals = 68;
__device__ __forceinline__ int walk_occurrences(const int32_t* __restrict__ tok, int64_t hi, const int32_t* __restrict__ h, int hl,
                                                uint32_t e0, uint32_t e1, bool a0, bool a1, int len, int K, int lane, int32_t* s_cur,
                                                int32_t* s_val) {
  auto next = [&](uint32_t e, int j) -> int32_t {
    if (e & 0x80000000u) {
      const int idx = int(e & 0x7fffffffu) + j;
      return idx < hl ? h[idx] : -1;
    }
    const int64_t p = int64_t(e) + j;
    return p < hi ? tok[p] : -1;
  };
  auto of_depth = [](const int32_t (&r)[kWalkDepths], int u) {    // (the loop over the depths is not unrolled: half the code)
    int32_t t = r[0];
#pragma unroll
    for (int x = 1; x < kWalkDepths; ++x) t = u == x ? r[x] : t;
    return t;
  };
  const unsigned below = (1u << lane) - 1;
  constexpr int32_t kNone = 0x7fffffff;
  __syncwarp();                         // (s_val may be where e0 and e1 came from)
  while (len < K) {
    unsigned m0 = __ballot_sync(0xffffffffu, a0), m1 = __ballot_sync(0xffffffffu, a1);
    int c = __popc(m0) + __popc(m1);
    if (c == 0) break;
    if (c <= kWalkFew) {
      const int base = len;             // of the 32 depths that the lanes hold
      int32_t x[kWalkFew];
      unsigned l0 = m0, l1 = m1, left = (1u << c) - 1;
#pragma unroll
      for (int i = 0; i < kWalkFew; ++i) {
        x[i] = -1;
        if (i >= c) continue;           // (uniform)
        const uint32_t e = __shfl_sync(0xffffffffu, l0 ? e0 : e1, __ffs(l0 ? l0 : l1) - 1);
        if (l0) l0 &= l0 - 1; else l1 &= l1 - 1;
        if (base + 1 + lane <= K) x[i] = next(e, base + 1 + lane);
      }
      while (left) {
        int32_t v = -1;
        bool same = true;
#pragma unroll
        for (int i = kWalkFew - 1; i >= 0; --i) if (left >> i & 1u) v = x[i];
#pragma unroll
        for (int i = 0; i < kWalkFew; ++i) same = same && (!(left >> i & 1u) || x[i] == v);
        const unsigned part = __ballot_sync(0xffffffffu, !same || v < 0) & (~0u << (len - base));
        const int d = part ? __ffs(part) - 1 : 32;
        if (lane >= len - base && lane < d) s_cur[base + lane] = v;
        len = base + d;
        if (d == 32 || len >= K) break;
        // lane d holds the tokens of the depth at which they part or end; lane i votes for the i-th
        int32_t mine = -1;
        int votes = 0;
        int32_t y[kWalkFew];
#pragma unroll
        for (int i = 0; i < kWalkFew; ++i) {
          y[i] = __shfl_sync(0xffffffffu, x[i], d);
          if (!(left >> i & 1u)) y[i] = -1;
          if (lane == i) mine = y[i];
        }
#pragma unroll
        for (int i = 0; i < kWalkFew; ++i) votes += y[i] == mine;
        if (mine < 0) votes = 0;
        const int best = __reduce_max_sync(0xffffffffu, votes);
        const int32_t pick = __reduce_min_sync(0xffffffffu, votes == best ? mine : kNone);
        left = best ? __ballot_sync(0xffffffffu, votes > 0 && mine == pick) : 0u;
        if (!left) break;
        if (lane == 0) s_cur[len] = pick;
        if (++len >= K || len - base == 32) break;
      }
      if (!left) break;
      a0 = a0 && (left >> __popc(m0 & below) & 1u);
      a1 = a1 && (left >> (__popc(m0) + __popc(m1 & below)) & 1u);
      continue;
    }
    int32_t r0[kWalkDepths], r1[kWalkDepths];
#pragma unroll
    for (int u = 0; u < kWalkDepths; ++u) {
      r0[u] = a0 && len + 1 + u <= K ? next(e0, len + 1 + u) : -1;
      r1[u] = a1 && len + 1 + u <= K ? next(e1, len + 1 + u) : -1;
    }
#pragma unroll 1
    for (int u = 0; u < kWalkDepths && len < K; ++u) {
      const int32_t t0 = of_depth(r0, u);
      const int32_t t1 = of_depth(r1, u);
      a0 = a0 && t0 >= 0; a1 = a1 && t1 >= 0;
      m0 = __ballot_sync(0xffffffffu, a0); m1 = __ballot_sync(0xffffffffu, a1);
      c = __popc(m0) + __popc(m1);
      if (c <= 1) break;
      const int32_t first = __shfl_sync(0xffffffffu, m0 ? t0 : t1, __ffs(m0 ? m0 : m1) - 1);
      if (2 * (__popc(__ballot_sync(0xffffffffu, a0 && t0 == first)) + __popc(__ballot_sync(0xffffffffu, a1 && t1 == first))) > c) {
        a0 = a0 && t0 == first; a1 = a1 && t1 == first;
        if (lane == 0) s_cur[len] = first;
        ++len;
        continue;
      }
      if (a0) s_val[__popc(m0 & below)] = t0;
      if (a1) s_val[__popc(m0) + __popc(m1 & below)] = t1;
      if (lane < 4) s_val[c + lane] = -1;
      __syncwarp();
      int n0 = 0, n1 = 0;
#pragma unroll 4
      for (int j = 0; j < c; j += 4) {
        const int4 w = *reinterpret_cast<const int4*>(s_val + j);
        n0 += (w.x == t0) + (w.y == t0) + (w.z == t0) + (w.w == t0);
        n1 += (w.x == t1) + (w.y == t1) + (w.z == t1) + (w.w == t1);
      }
      n0 = a0 ? n0 : 0; n1 = a1 ? n1 : 0;
      const int best = __reduce_max_sync(0xffffffffu, max(n0, n1));
      const int32_t pick = __reduce_min_sync(0xffffffffu, min(n0 == best ? t0 : kNone, n1 == best ? t1 : kNone));
      a0 = a0 && t0 == pick; a1 = a1 && t1 == pick;
      if (lane == 0) s_cur[len] = pick;
      ++len;
      __syncwarp();                     // (s_val is read)
    }
  }
  __syncwarp();
  return len;
}

constexpr int kDraftWarps = 4;
// Work list of the large-run kernel: runs that a team of it holds and longer ones, the next of each, CTAs done; then (query, suffix
// length, start of its run), of the former from the front and of the latter from the back.
enum { WORK_SHORT = 0, WORK_LONG, WORK_NEXT_SHORT, WORK_NEXT_LONG, WORK_DONE, WORK_HEAD };
constexpr int kTeamRun = 2048; // positions of the longest run that a team takes

// The first probes of four suffix lengths, n and below, at once: eight lanes and slots each, from the keys' home slots on.  A bit
// per length: settled (found, or an empty slot seen first: not there) and found, then `off` in that length's first lane is the
// slot's distance from home.  A length after the other is a round trip to memory each, of the ten or so that a query takes.
constexpr int kProbeLevels = 4, kProbeLanes = 32 / kProbeLevels;
struct FirstProbe { unsigned settled, found; uint32_t off; };
__device__ __forceinline__ FirstProbe probe_first(const PoolView& pv, const DraftArgs& a, const Region& rg, int q, int g, int n, int lane) {
  const int mine = n - lane / kProbeLanes;
  const uint32_t slot = lane % kProbeLanes;
  uint64_t key = key_begin(g, mine);
  bool there = mine >= a.n_min;
  for (int j = 0; j < mine; ++j) {
    const int32_t t = a.tails[size_t(q) * a.n_max + a.n_max - mine + j];
    there = there && t >= 0;
    key = key_push(key, t);
  }
  key = key_end(key);
  uint2 e = make_uint2(0xffffffffu, 0xffffffffu);
  if (there) {
    uint64_t s = uint64_t(home_slot(key, rg.slots)) + slot;   // (a small region is seen more than once, as in probe)
    if (s >= rg.slots) s %= rg.slots;
    e = __ldg(pv.table[mine] + rg.base + s);
  }
  const unsigned empty = __ballot_sync(0xffffffffu, e.y == 0xffffffffu), hit = __ballot_sync(0xffffffffu, e.y != 0xffffffffu && e.x == uint32_t(key));
  const unsigned shift = lane / kProbeLanes * kProbeLanes, em = empty >> shift & ((1u << kProbeLanes) - 1);
  unsigned hm = hit >> shift & ((1u << kProbeLanes) - 1);
  if (em) hm &= (em & -em) - 1u;
  FirstProbe r;
  r.off = hm ? uint32_t(__ffs(hm) - 1) : 0u;
  const unsigned settled = __ballot_sync(0xffffffffu, (em || hm) && slot == 0), found = __ballot_sync(0xffffffffu, hm && slot == 0);
  r.settled = r.found = 0;
#pragma unroll
  for (int x = 0; x < kProbeLevels; ++x) {
    r.settled |= (settled >> (x * kProbeLanes) & 1u) << x;
    r.found |= (found >> (x * kProbeLanes) & 1u) << x;
  }
  return r;
}

__global__ void __launch_bounds__(kDraftWarps * 32)
draft_warp_kernel(PoolView pv, DraftArgs a) {
  __shared__ __align__(16) uint32_t s_occ[kDraftWarps][kWalkVals];   // occurrences, then the walk's
  __shared__ int32_t s_cur[kDraftWarps][kMaxK];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int q = blockIdx.x * kDraftWarps + warp;
  next_may_launch();
  if (q >= a.B) return;
  wait_for_earlier();
  int32_t* out = a.draft + size_t(q) * a.K;
  const int g = a.group_id[q];
  int best_len = 0, best_n = 0;
  int overflow = 0;                  // suffix length from which the large-run kernel takes over, where its run starts,
  uint32_t start = 0;
  bool big = false;                  // and whether a team of that kernel cannot hold it
  if (g >= 0 && g < pv.G) {
    const int64_t lo = pv.goff[g], hi = pv.goff[g + 1];
    const int tl = min(max(a.tail_len[q], 0), a.n_max);
    const Region rg = region_of(lo, hi, g);
    FirstProbe fp{};
    for (int n = tl, base = 0; n >= a.n_min && !overflow; --n) {
      if (n == tl || n == base - kProbeLevels) { base = n; fp = probe_first(pv, a, rg, q, g, n, lane); }
      const int level = base - n;
      if (fp.settled >> level & ~(fp.found >> level) & 1u) continue;   // not there
      int32_t tn[kMaxN];  // the last n tail tokens, oldest first
      uint64_t h = key_begin(g, n);
      for (int j = 0; j < n; ++j) {
        tn[j] = a.tails[size_t(q) * a.n_max + a.n_max - n + j];
        h = key_push(h, tn[j]);
      }
      uint32_t off = (fp.found >> level & 1u) ? __shfl_sync(0xffffffffu, fp.off, level * kProbeLanes) : uint32_t(kProbeLanes);
      const int want = (a.max_occ > 0 && a.max_occ <= 64) ? a.max_occ : 65;
      int n_occ = gather_occurrences(pv, lo, hi, tn, n, key_end(h), g, lane, s_occ[warp], 0, want, start, off);
      if (want == 65 && n_occ > 64) {
        overflow = n;
        const int64_t last = int64_t(start) + kTeamRun;     // (a run is of one n-gram: a position of it there tells how long it is)
        big = (a.max_occ == 0 || a.max_occ > kTeamRun) && last < a.n_positions && is_occurrence(pv.tok, lo, hi, int64_t(pv.positions[n][last] & ~kRunEnd), tn, n);
        break;
      }
      n_occ = min(n_occ, min(want, 64));
      if (n_occ == 0) continue;
      __syncwarp();
      const int len = walk_occurrences(pv.tok, hi, nullptr, 0, lane < n_occ ? s_occ[warp][lane] : 0u,
                                       lane + 32 < n_occ ? s_occ[warp][lane + 32] : 0u, lane < n_occ, lane + 32 < n_occ, 0, a.K, lane, s_cur[warp],
                                       reinterpret_cast<int32_t*>(s_occ[warp]));
      if (len > best_len) {
        for (int j = lane; j < len; j += 32) out[j] = s_cur[warp][j];
        best_len = len; best_n = n;
      }
      __syncwarp();
      if (best_len >= max(a.min_draft, 1)) break;
    }
  }
  if (overflow) {  // the rest of the query, and the best draft so far, to the large-run kernel
    if (lane == 0) {
      const int at = atomicAdd(&a.work[big ? WORK_LONG : WORK_SHORT], 1);
      int32_t* w = a.work + WORK_HEAD + 3 * (big ? a.B - 1 - at : at);
      w[0] = q; w[1] = overflow; w[2] = int32_t(start);
      a.draft_len[q] = best_len; a.match_n[q] = best_n;
    }
    return;
  }
  for (int j = best_len + lane; j < a.K; j += 32) out[j] = -1;
  if (lane == 0) { a.draft_len[q] = best_len; a.match_n[q] = best_len ? best_n : 0; }
}

// Temporary branches (Section 3.2): the same retrieval with the sequence's own text (prompt +
// generated tokens) searched as one more document.  Its occurrences of the tail that still have
// a following token come first in the occurrence list, the group's follow, and the list is cut
// to max_occ (1..64).  An occurrence is tagged with bit 31 when it lies in the history.
struct TempArgs {
  const int32_t* hist; const int32_t* hist_len; int64_t hist_stride;
};

__global__ void __launch_bounds__(kDraftWarps * 32)
draft_temp_kernel(PoolView pv, DraftArgs a, TempArgs t) {
  __shared__ __align__(16) uint32_t s_occ[kDraftWarps][kWalkVals];   // occurrences, then the walk's
  __shared__ int32_t s_cur[kDraftWarps][kMaxK];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int q = blockIdx.x * kDraftWarps + warp;
  next_may_launch();
  if (q >= a.B) return;
  wait_for_earlier();
  int32_t* out = a.draft + size_t(q) * a.K;
  const int g = a.group_id[q];
  const bool has_group = g >= 0 && g < pv.G;
  const int64_t lo = has_group ? pv.goff[g] : 0, hi = has_group ? pv.goff[g + 1] : 0;
  const int32_t* h = t.hist + size_t(q) * t.hist_stride;
  const int hl = max(t.hist_len[q], 0);
  const int cap = a.max_occ;
  int best_len = 0, best_n = 0;
  const int tl = min(max(a.tail_len[q], 0), a.n_max);
  for (int n = tl; n >= a.n_min; --n) {
    int32_t tn[kMaxN];  // the last n tail tokens, oldest first
    bool bad = false;
    uint64_t key = key_begin(g, n);
    for (int j = 0; j < n; ++j) {
      tn[j] = a.tails[size_t(q) * a.n_max + a.n_max - n + j];
      bad |= tn[j] < 0;
      key = key_push(key, tn[j]);
    }
    if (bad) continue;
    int n_occ = 0;
    for (int base = 0; base + 1 < hl && n_occ < cap; base += 32) {   // the history, ascending
      const int idx = base + lane;
      bool ok = idx >= n - 1 && idx + 1 < hl;
      for (int j = 0; ok && j < n; ++j) ok = h[idx - n + 1 + j] == tn[j];
      const unsigned ball = __ballot_sync(0xffffffffu, ok);
      const int slot = n_occ + __popc(ball & ((1u << lane) - 1));
      if (ok && slot < 64) s_occ[warp][slot] = uint32_t(idx) | 0x80000000u;
      n_occ += __popc(ball);
    }
    n_occ = min(n_occ, cap);
    uint32_t start;
    if (has_group && n_occ < cap)   // the group, ascending
      n_occ = min(cap, gather_occurrences(pv, lo, hi, tn, n, key_end(key), g, lane, s_occ[warp], n_occ, cap, start));
    if (n_occ == 0) continue;
    __syncwarp();
    const int len = walk_occurrences(pv.tok, hi, h, hl, lane < n_occ ? s_occ[warp][lane] : 0u, lane + 32 < n_occ ? s_occ[warp][lane + 32] : 0u,
                                     lane < n_occ, lane + 32 < n_occ, 0, a.K, lane, s_cur[warp],
                                       reinterpret_cast<int32_t*>(s_occ[warp]));
    if (len > best_len) {
      for (int j = lane; j < len; j += 32) out[j] = s_cur[warp][j];
      best_len = len; best_n = n;
    }
    __syncwarp();
    if (best_len >= max(a.min_draft, 1)) break;
  }
  for (int j = best_len + lane; j < a.K; j += 32) out[j] = -1;
  if (lane == 0) { a.draft_len[q] = best_len; a.match_n[q] = best_len ? best_n : 0; }
}

// Tree-based drafting (Section 3.3): the sub-tree under the matched tail, cut to its K most
// frequent nodes, listed depth-first.  One warp per query.  The occurrences (history first if
// given, then the group's, at most max_occ <= 64) each carry a continuation of up to K tokens; a
// trie node is a pair (occurrence o, depth d) = the first d tokens of o's continuation, owned by
// the first occurrence that has that prefix.  Pairwise common-prefix lengths give every node's
// frequency; nodes are taken best first by (frequency descending, depth ascending, token path
// ascending) -- along one occurrence that is by increasing depth, so each occurrence offers one
// candidate per round -- and the kept nodes are ranked into depth-first order, children by
// (frequency descending, token ascending).
constexpr int kTreeK = 32;   // nodes of a drafted tree (one lane ranks one node)

__global__ void __launch_bounds__(32)
draft_tree_kernel(PoolView pv, DraftArgs a, TempArgs t, int32_t* __restrict__ draft_parents) {
  __shared__ uint32_t s_occ[64];
  __shared__ int32_t s_cont[64][kTreeK];
  __shared__ uint8_t s_len[64], s_own[64];         // continuation length; first depth the occurrence owns
  __shared__ uint8_t s_lcp[64][64];
  __shared__ uint8_t s_freq[64][kTreeK];           // frequency of node (o, d) at [o][d-1]
  __shared__ int s_sel_o[kTreeK], s_sel_d[kTreeK], s_rank[kTreeK];
  const int lane = threadIdx.x, q = blockIdx.x;
  next_may_launch();
  if (q >= a.B) return;
  wait_for_earlier();
  int32_t* out = a.draft + size_t(q) * a.K;
  int32_t* outp = draft_parents + size_t(q) * a.K;
  const int K = a.K;
  const int g = a.group_id[q];
  const bool has_group = g >= 0 && g < pv.G;
  const int64_t lo = has_group ? pv.goff[g] : 0, hi = has_group ? pv.goff[g + 1] : 0;
  const int32_t* h = t.hist ? t.hist + size_t(q) * t.hist_stride : nullptr;
  const int hl = t.hist ? max(t.hist_len[q], 0) : 0;
  const int cap = a.max_occ;
  int best_len = 0, best_n = 0;
  const int tl = min(max(a.tail_len[q], 0), a.n_max);
  for (int n = tl; n >= a.n_min; --n) {
    int32_t tn[kMaxN];
    bool bad = false;
    uint64_t key = key_begin(g, n);
    for (int j = 0; j < n; ++j) {
      tn[j] = a.tails[size_t(q) * a.n_max + a.n_max - n + j];
      bad |= tn[j] < 0;
      key = key_push(key, tn[j]);
    }
    if (bad) continue;
    // ---- occurrences ----
    int n_occ = 0;
    for (int base = 0; base + 1 < hl && n_occ < cap; base += 32) {
      const int idx = base + lane;
      bool ok = idx >= n - 1 && idx + 1 < hl;
      for (int j = 0; ok && j < n; ++j) ok = h[idx - n + 1 + j] == tn[j];
      const unsigned ball = __ballot_sync(0xffffffffu, ok);
      const int slot = n_occ + __popc(ball & ((1u << lane) - 1));
      if (ok && slot < 64) s_occ[slot] = uint32_t(idx) | 0x80000000u;
      n_occ += __popc(ball);
    }
    n_occ = min(n_occ, cap);
    uint32_t start;
    if (has_group && n_occ < cap) n_occ = min(cap, gather_occurrences(pv, lo, hi, tn, n, key_end(key), g, lane, s_occ, n_occ, cap, start));
    if (n_occ == 0) continue;
    __syncwarp();
    // ---- continuations ----
    for (int o = lane; o < n_occ; o += 32) {
      const uint32_t e = s_occ[o];
      int len = 0;
      for (int j = 1; j <= K; ++j) {
        int32_t tok;
        if (e & 0x80000000u) { const int idx = int(e & 0x7fffffffu) + j; tok = idx < hl ? h[idx] : -1; }
        else { const int64_t p = int64_t(e) + j; tok = p < hi ? pv.tok[p] : -1; }
        if (tok < 0) break;
        s_cont[o][len++] = tok;
      }
      s_len[o] = uint8_t(len);
    }
    __syncwarp();
    // ---- pairwise common-prefix lengths ----
    for (int pr = lane; pr < n_occ * n_occ; pr += 32) {
      const int o = pr / n_occ, o2 = pr % n_occ;
      const int lim = min(int(s_len[o]), int(s_len[o2]));
      int l = 0;
      while (l < lim && s_cont[o][l] == s_cont[o2][l]) ++l;
      s_lcp[o][o2] = uint8_t(l);
    }
    __syncwarp();
    // ---- node frequencies; the depth from which an occurrence owns its nodes ----
    for (int o = lane; o < n_occ; o += 32) {
      uint8_t hist_l[kTreeK + 1];
      for (int d = 0; d <= K; ++d) hist_l[d] = 0;
      int shared_before = 0;
      for (int o2 = 0; o2 < n_occ; ++o2) {
        const int l = s_lcp[o][o2];
        ++hist_l[l];
        if (o2 < o) shared_before = max(shared_before, l);
      }
      int run = 0;
      for (int d = int(s_len[o]); d >= 1; --d) { run += hist_l[d]; s_freq[o][d - 1] = uint8_t(run); }
      s_own[o] = uint8_t(shared_before + 1);
    }
    __syncwarp();
    // ---- best-first selection: each occurrence offers its shallowest untaken own node ----
    int nd0 = lane < n_occ ? int(s_own[lane]) : 255, nd1 = lane + 32 < n_occ ? int(s_own[lane + 32]) : 255;
    int m = 0;
    auto pack = [&](int o, int d) -> unsigned {   // smaller = better; ties are resolved by the token path below
      const unsigned f = s_freq[o][d - 1];
      return ((255u - f) << 16) | (unsigned(d) << 8) | unsigned(o);
    };
    auto path_less = [&](int o, int o2, int d) -> bool {   // same frequency and depth, different nodes
      const int l = s_lcp[o][o2];
      return s_cont[o][l] < s_cont[o2][l];
    };
    auto node_better = [&](unsigned x, unsigned y) -> bool {
      if (y == 0xffffffffu) return x != 0xffffffffu;
      if (x == 0xffffffffu) return false;
      if ((x >> 8) != (y >> 8)) return (x >> 8) < (y >> 8);
      const int o = int(x & 255u), o2 = int(y & 255u), d = int((x >> 8) & 255u);
      if (o == o2) return false;
      return path_less(o, o2, d);
    };
    while (m < K) {
      unsigned c0 = (nd0 <= (lane < n_occ ? int(s_len[lane]) : 0)) ? pack(lane, nd0) : 0xffffffffu;
      const unsigned c1 = (nd1 <= (lane + 32 < n_occ ? int(s_len[lane + 32]) : 0)) ? pack(lane + 32, nd1) : 0xffffffffu;
      if (node_better(c1, c0)) c0 = c1;
      for (int off = 16; off; off >>= 1) {
        const unsigned other = __shfl_xor_sync(0xffffffffu, c0, off);
        if (node_better(other, c0)) c0 = other;
      }
      if (c0 == 0xffffffffu) break;
      const int o = int(c0 & 255u), d = int((c0 >> 8) & 255u);
      if (lane == 0) { s_sel_o[m] = o; s_sel_d[m] = d; }
      if (o == lane) ++nd0;
      if (o == lane + 32) ++nd1;
      ++m;
    }
    __syncwarp();
    if (m > best_len) {
      // ---- depth-first rank of every kept node (lane k ranks node k) ----
      int rank = 0;
      const int ok_ = lane < m ? s_sel_o[lane] : 0, dk = lane < m ? s_sel_d[lane] : 0;
      if (lane < m) {
        for (int j = 0; j < m; ++j) {
          if (j == lane) continue;
          const int oj = s_sel_o[j], dj = s_sel_d[j];
          const int l = min(int(s_lcp[oj][ok_]), min(dj, dk));
          bool before;
          if (l == dj) before = true;                 // j is an ancestor of this node
          else if (l == dk) before = false;           // this node is an ancestor of j
          else {                                      // they part at depth l + 1: compare those siblings
            const int fj = s_freq[oj][l], fk = s_freq[ok_][l];
            before = fj > fk || (fj == fk && s_cont[oj][l] < s_cont[ok_][l]);
          }
          rank += before;
        }
        s_rank[lane] = rank;
      }
      __syncwarp();
      if (lane < m) {
        int parent_row = 0;
        if (dk > 1)
          for (int j = 0; j < m; ++j)
            if (s_sel_d[j] == dk - 1 && int(s_lcp[s_sel_o[j]][ok_]) >= dk - 1) { parent_row = s_rank[j] + 1; break; }
        out[rank] = s_cont[ok_][dk - 1];
        outp[rank] = parent_row;
      }
      best_len = m; best_n = n;
    }
    __syncwarp();
    if (best_len >= max(a.min_draft, 1)) break;
  }
  for (int j = best_len + lane; j < K; j += 32) { out[j] = -1; outp[j] = -1; }
  if (lane == 0) { a.draft_len[q] = best_len; a.match_n[q] = best_len ? best_n : 0; }
}

__global__ void make_tree_rows_kernel(const int32_t* last, const int32_t* draft, const int32_t* dpar, const int32_t* dlen, int B, int K,
                                      int32_t* tokens, int32_t* parents, int32_t* n_rows, unsigned long long* stamp) {
  next_may_launch();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B * (K + 1)) return;
  const int b = i / (K + 1), j = i % (K + 1);
  wait_for_earlier();
  const int32_t lt = last[b];
  const int m = lt < 0 ? 0 : min(max(dlen[b], 0), K);
  tokens[i] = lt < 0 ? -1 : (j == 0 ? lt : (j <= m ? draft[b * K + j - 1] : -1));
  parents[i] = (lt >= 0 && j >= 1 && j <= m) ? dpar[b * K + j - 1] : -1;
  if (j == 0) n_rows[b] = lt < 0 ? 0 : 1 + m;
  if (stamp && i == 0) *stamp = device_ns();
}

// Large-run path.  Runs of up to 2048 positions - nearly all of them - go to teams of 256 threads, four a CTA, that hold the run's
// positions in registers and vote through a small hash table in shared memory; longer ones, first, to whole CTAs that hold
// 16384 and vote in a histogram over the vocabulary.  The warp kernel passes on where the run starts and which of the two it is
// for; what does not fit after all, and the shorter suffixes of a query whose draft is too short, are left to the CTA.
// Such a run is read once: its occurrences (those whose tokens match the tail) vote on the first token while their
// positions go to a list in shared memory; from then on only the list is walked, cut after every vote to the occurrences
// that continue with the winner - a small share of them, as token frequencies fall fast.  A run that overflows the list is
// read again at every depth, with the draft so far compared, until what is left fits.  Up to 64 survivors are walked by one
// warp in registers.
// Bound by the latency of the longest run's chain of loads.  4096 queries on 50 M tokens in 10,000 groups - about 210 have such
// runs, a dozen of them long - the warp kernel included: 62 us a batch with all of them served by whole CTAs that read the
// run and then a list, 51 with these, 34 with the walk by lanes of depths.  Where max_occ cuts the runs (500, groups of 25 k tokens, 300
// queries) 31 and 26.
constexpr int kBigThreads = 1024;
constexpr int kBigUnroll = 4;
constexpr int kBigList = 4096;      // positions: four a thread

// A run held in registers by THREADS threads of a CTA (whose barrier is number `bar`), ITEMS positions each: the query's run of suffix
// length n from `start` on.  Votes go to a histogram over the vocabulary (HIST: all zero before and after), or to a hash table
// of {token | votes}, 16 bits each.  0: done; else the suffix length from which the CTA goes on - n itself where the run is too
// long - with the draft so far in place.
constexpr int kTeams = 4, kTeamThreads = kBigThreads / kTeams, kTeamItems = kTeamRun / kTeamThreads;
constexpr int kTeamSlots = 2 * kTeamRun, kTeamSlotBits = 12;
constexpr int kLongItems = 16;
static_assert(kTeamItems * kTeamThreads == kTeamRun && kTeamSlots == 1 << kTeamSlotBits && kTeamRun < 65536, "");
// Shared memory for the histogram and a longer list, as far as the vocabulary leaves room, where max_occ does not bound the list; otherwise
// what the teams' tables take.  A longer list spares passes over the run, and what it takes is lost to the L1 cache, in which the
// occurrences' next tokens wait for the depths to come.  Groups of 200 thousand tokens: max_occ 500, 512 queries 32.6 us with the longer
// list, 30.5 without, of min_draft 8 48.2 and 45.3; max_occ 0 286 and 379 (runs of 49 and 109 thousand), but 64 queries of
// which one has a run of 31 thousand 127 and 107.
constexpr size_t kHistMost = 200 * 1024, kBigSmem = 204 * 1024, kTeamSmem = size_t(kTeams) * kTeamSlots * sizeof(uint32_t);
static_assert(kTeamSmem <= kBigSmem && kBigSmem <= kHistMost + kBigList * sizeof(uint32_t), "");
struct Held {
  __align__(16) uint32_t list[kWalkVals];   // occurrences, then the walk's
  uint32_t end, count;
  unsigned long long best;
  int item[3], reached, odd;    // odd: a position that does not match
  int32_t cur[kMaxK];
};

template <int THREADS, int ITEMS, bool HIST>
__device__ __forceinline__ int held_run(const PoolView& pv, const DraftArgs& a, Held& s, uint32_t* table, int bar, int q, int n,
                                        uint32_t start) {
  const int tt = threadIdx.x % THREADS, lane = tt & 31, warp = tt >> 5;
  auto barrier = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(THREADS) : "memory"); };
  // Where max_occ occurrences are all that count, the run's first max_occ positions are those: they are if all of them match.
  const bool cut = a.max_occ > 0 && a.max_occ <= THREADS * ITEMS;
  const int most = cut ? a.max_occ : THREADS * ITEMS;
  const uint32_t* plist = pv.positions[n] + start;
  uint32_t v[ITEMS], alive = 0;                    // positions; a bit for each that counts
  uint32_t end = 0xffffffffu;
#pragma unroll
  for (int u = 0; u < ITEMS; ++u) {
    const int idx = u * THREADS + tt;
    v[u] = idx < most ? (int64_t(start) + idx < a.n_positions ? plist[idx] : kRunEnd) : 0u;
  }
#pragma unroll
  for (int u = ITEMS - 1; u >= 0; --u) if (v[u] & kRunEnd) end = uint32_t(u * THREADS + tt);
  const int g = a.group_id[q];
  const int64_t lo = pv.goff[g], hi = pv.goff[g + 1];
  int32_t tn[kMaxN];
  for (int j = 0; j < n; ++j) tn[j] = a.tails[size_t(q) * a.n_max + a.n_max - n + j];
  if (tt == 0) { s.end = 0xffffffffu; s.odd = 0; s.best = 0; s.count = 0; }
  if (!HIST) for (int x = tt; x < kTeamSlots; x += THREADS) table[x] = 0xffffffffu;
  barrier();
  end = __reduce_min_sync(0xffffffffu, end);
  if (lane == 0 && end != 0xffffffffu) atomicMin(&s.end, end);
  barrier();
  const bool whole = s.end != 0xffffffffu;
  if (!whole && !cut) return n;
  end = whole ? s.end : uint32_t(most) - 1;
  int32_t t[ITEMS];
  bool odd = false;
#pragma unroll
  for (int u = 0; u < ITEMS; ++u) {
    t[u] = -1;
    if (uint32_t(u * THREADS + tt) > end) continue;
    if (occurrence_and_next(pv.tok, lo, hi, int64_t(v[u] & ~kRunEnd), tn, n, 1, t[u])) alive |= 1u << u;
    else odd = true;
  }
  if (!whole) {
    if (odd) s.odd = 1;
    barrier();
    if (s.odd) return n;
  }
  const int best_len = a.draft_len[q];             // of the longer suffixes, with their draft in place
  int len = 0;
  for (;;) {                                       // t: the tokens of depth len + 1
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) if (t[u] < 0) alive &= ~(1u << u);
    const uint32_t left = __reduce_add_sync(0xffffffffu, uint32_t(__popc(alive)));
    if (lane == 0 && left) atomicAdd(&s.count, left);
    barrier();
    const uint32_t count = s.count;
    barrier();
    if (tt == 0) { s.count = 0; s.best = 0; }
    barrier();
    if (count <= 64) {                             // one warp walks them
#pragma unroll
      for (int u = 0; u < ITEMS; ++u) if (alive >> u & 1u) s.list[atomicAdd(&s.count, 1u)] = v[u] & ~kRunEnd;
      barrier();
      if (warp == 0) {
        const int l = count ? walk_occurrences(pv.tok, hi, nullptr, 0, lane < count ? s.list[lane] : 0u, lane + 32 < count ? s.list[lane + 32] : 0u,
                                               lane < count, lane + 32 < count, len, a.K, lane, s.cur,
                                               reinterpret_cast<int32_t*>(s.list)) : len;
        if (lane == 0) s.reached = l;
      }
      barrier();
      len = s.reached;
      break;
    }
    unsigned long long cand = 0;
    uint32_t at[HIST ? 1 : ITEMS];
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
      if (!(alive >> u & 1u)) continue;
      uint32_t votes;                              // whoever votes last sees the token's full count
      if (HIST) {
        votes = atomicAdd(table + t[u], 1u) + 1;
      } else {
        uint32_t x = (uint32_t(t[u]) * 0x9E3779B1u) >> (32 - kTeamSlotBits);
        for (;; x = (x + 1) & (kTeamSlots - 1)) {  // (there are more slots than positions)
          uint32_t w = *const_cast<volatile uint32_t*>(table + x);
          if (w == 0xffffffffu) {
            w = atomicCAS(table + x, 0xffffffffu, uint32_t(t[u]) << 16 | 1u);
            if (w == 0xffffffffu) { votes = 1; break; }
          }
          if (w >> 16 == uint32_t(t[u])) { votes = (atomicAdd(table + x, 1u) & 0xffffu) + 1; break; }
        }
        at[HIST ? 0 : u] = x;
      }
      cand = max(cand, (unsigned long long)((uint64_t(votes) << 32) | uint32_t(0x7fffffff - t[u])));
    }
    for (int o = 16; o; o >>= 1) cand = max(cand, __shfl_xor_sync(0xffffffffu, cand, o));
    if (lane == 0 && cand) atomicMax(&s.best, cand);
    barrier();
    const int32_t pick = 0x7fffffff - int32_t(uint32_t(s.best));
    if (tt == 0) s.cur[len] = pick;
    ++len;
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
      if (!(alive >> u & 1u)) continue;
      table[HIST ? uint32_t(t[u]) : at[HIST ? 0 : u]] = HIST ? 0u : 0xffffffffu;
      if (t[u] != pick) { alive &= ~(1u << u); continue; }
      const int64_t p = int64_t(v[u] & ~kRunEnd) + len + 1;
      t[u] = p < hi && len < a.K ? pv.tok[p] : -1;
    }
    if (len == a.K) break;
  }
  barrier();                                       // (s.cur is complete)
  int32_t* out = a.draft + size_t(q) * a.K;
  const bool better = len > best_len, done = max(len, best_len) >= max(a.min_draft, 1) || n == a.n_min;
  if (better) for (int j = tt; j < len; j += THREADS) out[j] = s.cur[j];
  if (done) for (int j = max(len, best_len) + tt; j < a.K; j += THREADS) out[j] = -1;
  if (tt == 0 && better) { a.draft_len[q] = len; a.match_n[q] = n; }
  if (tt == 0 && !better && best_len == 0) a.match_n[q] = 0;
  return done ? 0 : n - 1;
}

__global__ void __launch_bounds__(kBigThreads)
draft_cta_kernel(PoolView pv, DraftArgs a, int vocab_bound, uint32_t list_cap) {
  extern __shared__ uint32_t s_hist[];            // [vocab_bound] votes, all zero between depths; then the list; or the teams' tables
  uint32_t* s_list = s_hist + vocab_bound;
  __shared__ int32_t s_cur[kMaxK];
  __shared__ uint32_t s_start, s_off, s_end, s_cut, s_count;
  __shared__ int s_found, s_item, s_warp_n[kBigThreads / 32];
  __shared__ unsigned long long s_best;
  __shared__ __align__(16) int32_t s_walk[kWalkVals];
  __shared__ Held s_team[kTeams];
  __shared__ Held s_held;
  __shared__ int s_late[kTeams][2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  next_may_launch();
  for (int v = tid; v < vocab_bound; v += kBigThreads) s_hist[v] = 0;
  wait_for_earlier();

  // A query by the whole CTA, from suffix length n_first on.
  auto serve = [&](int q, int n_first) {
    int32_t* out = a.draft + size_t(q) * a.K;
    const int g = a.group_id[q];
    const int64_t lo = pv.goff[g], hi = pv.goff[g + 1];
    int best_len = a.draft_len[q], best_n = a.match_n[q];      // of the longer suffixes, with their draft in `out`
    for (int n = n_first; n >= a.n_min; --n) {
      int32_t tn[kMaxN];
      bool bad = false;
      uint64_t h = key_begin(g, n);
      for (int j = 0; j < n; ++j) {
        tn[j] = a.tails[size_t(q) * a.n_max + a.n_max - n + j];
        bad |= tn[j] < 0;
        h = key_push(h, tn[j]);
      }
      if (bad) continue;
      int len = 0;
      uint32_t total = 0;                          // verified occurrences of the run
      for (uint32_t off = 0; total == 0; ++off) {  // (a run of another key with the same low half has none)
        if (warp == 0) {
          uint32_t st = 0;
          const Region rg = region_of(lo, hi, g);
          const bool f = probe(pv.table[n] + rg.base, rg.slots, key_end(h), lane, off, st);
          if (lane == 0) { s_found = f; s_start = st; s_off = off; s_end = s_cut = 0xffffffffu; }
        }
        __syncthreads();
        if (!s_found) break;
        off = s_off;
        const uint32_t* plist = pv.positions[n] + s_start;
        if (a.max_occ > 0) {                       // the run counts up to its max_occ-th verified occurrence
          uint32_t seen = 0;
          for (uint32_t base = 0;; base += kBigThreads) {
            const uint32_t idx = base + tid;
            const int64_t left = a.n_positions - int64_t(s_start);
            const uint32_t v = int64_t(idx) < left ? plist[idx] : kRunEnd;
            if (v & kRunEnd) atomicMin(&s_end, idx);
            __syncthreads();
            const bool ok = idx <= s_end && int64_t(idx) < left && is_occurrence(pv.tok, lo, hi, int64_t(v & ~kRunEnd), tn, n);
            const unsigned ball = __ballot_sync(0xffffffffu, ok);
            if (lane == 0) s_warp_n[warp] = __popc(ball);
            __syncthreads();
            uint32_t rank = seen + __popc(ball & ((1u << lane) - 1)), all = seen;
            for (int w = 0; w < kBigThreads / 32; ++w) { if (w < warp) rank += s_warp_n[w]; all += s_warp_n[w]; }
            if (ok && rank + 1 == uint32_t(a.max_occ)) s_cut = idx;
            seen = all;
            const bool more = s_end == 0xffffffffu && seen < uint32_t(a.max_occ);
            __syncthreads();
            if (!more) break;
          }
          if (tid == 0) s_end = 0xffffffffu;
          __syncthreads();
        }
        const uint32_t cut = s_cut;
        // depth j = len + 1 by passes over the run, until the alive occurrences fit the list
        bool listed = false;
        for (;;) {
          const int j = len + 1;
          if (tid == 0) { s_count = 0; s_best = 0; s_end = 0xffffffffu; }
          __syncthreads();
          unsigned long long cand = 0;
          uint32_t n_ok = 0;
          for (uint32_t base = 0;; base += kBigThreads * kBigUnroll) {
            uint32_t v[kBigUnroll];
#pragma unroll
            for (int u = 0; u < kBigUnroll; ++u) {
              const uint32_t idx = base + u * kBigThreads + tid;
              v[u] = int64_t(s_start) + idx < a.n_positions ? plist[idx] : kRunEnd;
              if (v[u] & kRunEnd) atomicMin(&s_end, idx);
            }
            __syncthreads();
            const uint32_t end = s_end;
            int32_t t[kBigUnroll];
            bool alive[kBigUnroll];
#pragma unroll
            for (int u = 0; u < kBigUnroll; ++u) {
              const uint32_t idx = base + u * kBigThreads + tid;
              const int64_t p = int64_t(v[u] & ~kRunEnd);
              alive[u] = idx <= end && idx <= cut && int64_t(s_start) + idx < a.n_positions;
              t[u] = -1;
              if (alive[u]) alive[u] = occurrence_and_next(pv.tok, lo, hi, p, tn, n, j, t[u]);
              n_ok += alive[u];
              alive[u] = alive[u] && t[u] >= 0;
              for (int x = 1; x < j && alive[u]; ++x) alive[u] = pv.tok[p + x] == s_cur[x - 1];
            }
#pragma unroll
            for (int u = 0; u < kBigUnroll; ++u) {
              if (alive[u]) {
                const uint32_t votes = atomicAdd(&s_hist[t[u]], 1u) + 1;   // whoever votes last sees the token's full count
                cand = max(cand, (unsigned long long)((uint64_t(votes) << 32) | uint32_t(0x7fffffff - t[u])));
              }
              const unsigned ball = __ballot_sync(0xffffffffu, alive[u]);
              uint32_t at = 0;
              if (ball && lane == 0) at = atomicAdd(&s_count, uint32_t(__popc(ball)));
              at = __shfl_sync(0xffffffffu, at, 0) + __popc(ball & ((1u << lane) - 1));
              if (alive[u] && at < list_cap) s_list[at] = v[u] & ~kRunEnd;
            }
            if (end != 0xffffffffu || base + kBigThreads * kBigUnroll > cut) break;
            __syncthreads();   // (every thread has read s_end)
          }
          for (int o = 16; o; o >>= 1) cand = max(cand, __shfl_xor_sync(0xffffffffu, cand, o));
          if (lane == 0 && cand) atomicMax(&s_best, cand);
          const uint32_t verified = __syncthreads_count(n_ok > 0);
          if (len == 0) total = verified;
          if (s_best == 0) break;                 // nothing continues
          for (int x = tid; x < vocab_bound; x += kBigThreads) s_hist[x] = 0;
          if (tid == 0) s_cur[j - 1] = 0x7fffffff - int32_t(uint32_t(s_best));
          len = j;
          const uint32_t count = s_count;
          listed = count <= kBigList;
          __syncthreads();
          if (!listed && count <= list_cap && len < a.K) {   // a long list, cut to the winner's occurrences where it is
            const int32_t pick = s_cur[len - 1];
            if (tid == 0) s_count = 0;
            for (uint32_t base = 0; base < count; base += kBigThreads * kBigUnroll) {
              uint32_t mine[kBigUnroll];
              bool keep[kBigUnroll];
#pragma unroll
              for (int u = 0; u < kBigUnroll; ++u) {
                const uint32_t idx = base + u * kBigThreads + tid;
                mine[u] = idx < count ? s_list[idx] : 0u;
                keep[u] = idx < count && int64_t(mine[u]) + len < hi && pv.tok[int64_t(mine[u]) + len] == pick;
              }
              __syncthreads();       // (what is written comes from here or before)
#pragma unroll
              for (int u = 0; u < kBigUnroll; ++u) {
                const unsigned ball = __ballot_sync(0xffffffffu, keep[u]);
                uint32_t at = 0;
                if (ball && lane == 0) at = atomicAdd(&s_count, uint32_t(__popc(ball)));
                at = __shfl_sync(0xffffffffu, at, 0) + __popc(ball & ((1u << lane) - 1));
                if (keep[u]) s_list[at] = mine[u];
              }
            }
            __syncthreads();
            listed = s_count <= kBigList;
            __syncthreads();
          }
          if (listed || len == a.K) break;
        }
        // the list holds the positions alive before the last vote: keep the winner's, then go on with the list alone
        while (listed && len < a.K) {
          const int32_t pick = s_cur[len - 1];
          const uint32_t count = s_count;
          uint32_t mine[kBigList / kBigThreads];
          bool keep[kBigList / kBigThreads];
#pragma unroll
          for (int u = 0; u < kBigList / kBigThreads; ++u) {
            const uint32_t idx = u * kBigThreads + tid;
            mine[u] = idx < count ? s_list[idx] : 0u;
            keep[u] = idx < count && int64_t(mine[u]) + len < hi && pv.tok[int64_t(mine[u]) + len] == pick;
          }
          __syncthreads();
          if (tid == 0) { s_count = 0; s_best = 0; }
          __syncthreads();
          const int j = len + 1;
          unsigned long long cand = 0;
          int32_t t[kBigList / kBigThreads];
#pragma unroll
          for (int u = 0; u < kBigList / kBigThreads; ++u) {
            t[u] = keep[u] && int64_t(mine[u]) + j < hi ? pv.tok[int64_t(mine[u]) + j] : -1;
            keep[u] = t[u] >= 0;
            const unsigned ball = __ballot_sync(0xffffffffu, keep[u]);
            uint32_t at = 0;
            if (ball && lane == 0) at = atomicAdd(&s_count, uint32_t(__popc(ball)));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(ball & ((1u << lane) - 1));
            if (keep[u]) s_list[at] = mine[u];
          }
          __syncthreads();
          if (s_count <= 64) break;
#pragma unroll
          for (int u = 0; u < kBigList / kBigThreads; ++u)
            if (keep[u]) {
              const uint32_t votes = atomicAdd(&s_hist[t[u]], 1u) + 1;
              cand = max(cand, (unsigned long long)((uint64_t(votes) << 32) | uint32_t(0x7fffffff - t[u])));
            }
          for (int o = 16; o; o >>= 1) cand = max(cand, __shfl_xor_sync(0xffffffffu, cand, o));
          if (lane == 0 && cand) atomicMax(&s_best, cand);
          __syncthreads();
#pragma unroll
          for (int u = 0; u < kBigList / kBigThreads; ++u)
            if (keep[u]) s_hist[t[u]] = 0;
          if (tid == 0) s_cur[j - 1] = 0x7fffffff - int32_t(uint32_t(s_best));
          len = j;
          __syncthreads();
        }
        if (listed && len < a.K && s_count > 0) {   // up to 64 survivors, all of which have a token at depth len + 1
          if (warp == 0) {
            const uint32_t c = s_count;
            const int l = walk_occurrences(pv.tok, hi, nullptr, 0, lane < c ? s_list[lane] : 0u, lane + 32 < c ? s_list[lane + 32] : 0u,
                                           lane < c, lane + 32 < c, len, a.K, lane, s_cur, s_walk);
            if (lane == 0) s_found = l;
          }
          __syncthreads();
          len = s_found;
        }
      }
      if (len > best_len) {
        for (int j = tid; j < len; j += kBigThreads) out[j] = s_cur[j];
        best_len = len; best_n = n;
      }
      __syncthreads();
      if (best_len >= max(a.min_draft, 1)) break;
    }
    for (int j = best_len + tid; j < a.K; j += kBigThreads) out[j] = -1;
    if (tid == 0) { a.draft_len[q] = best_len; a.match_n[q] = best_len ? best_n : 0; }
  };

  const int n_long = a.work[WORK_LONG], n_short = a.work[WORK_SHORT];
  for (;;) {
    __syncthreads();
    if (tid == 0) s_item = n_long ? atomicAdd(&a.work[WORK_NEXT_LONG], 1) : 0;
    __syncthreads();
    if (s_item >= n_long) break;
    const int32_t* w = a.work + WORK_HEAD + 3 * (a.B - 1 - s_item);
    const int q = w[0], rest = held_run<kBigThreads, kLongItems, true>(pv, a, s_held, s_hist, 0, q, w[1], uint32_t(w[2]));
    __syncthreads();
    if (rest) serve(q, rest);
  }
  const int team = tid / kTeamThreads;
  uint32_t* const table = s_hist + team * kTeamSlots;
  for (bool again = true; again;) {                // until no team has left a query and the list is empty
    if (tid % kTeamThreads == 0) s_late[team][1] = 0;
    for (;;) {
      Held& s = s_team[team];
      asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(kTeamThreads) : "memory");
      if (tid % kTeamThreads == 0) {
        const int i = atomicAdd(&a.work[WORK_NEXT_SHORT], 1);
        const int32_t* w = a.work + WORK_HEAD + 3 * i;
        s.item[0] = i < n_short ? w[0] : -1; s.item[1] = i < n_short ? w[1] : 0; s.item[2] = i < n_short ? w[2] : 0;
      }
      asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(kTeamThreads) : "memory");
      const int q = s.item[0];
      if (q < 0) break;
      const int rest = held_run<kTeamThreads, kTeamItems, false>(pv, a, s, table, 1 + team, q, s.item[1], uint32_t(s.item[2]));
      if (rest) {                                  // (the team waits for its CTA, which goes on with this one)
        if (tid % kTeamThreads == 0) { s_late[team][0] = q; s_late[team][1] = rest; }
        break;
      }
    }
    __syncthreads();
    again = false;
    for (int x = 0; x < kTeams; ++x) {
      if (!s_late[x][1]) continue;
      if (!again) for (int v = tid; v < vocab_bound; v += kBigThreads) s_hist[v] = 0;
      again = true;
      __syncthreads();
      serve(s_late[x][0], s_late[x][1]);
    }
    __syncthreads();                               // (s_late is read, and the histogram is the teams' tables again)
  }
  // the last CTA leaves the work list empty for the next call
  if (tid == 0 && atomicAdd(&a.work[WORK_DONE], 1) == int(gridDim.x) - 1)
    for (int x = 0; x < WORK_HEAD; ++x) a.work[x] = 0;
}

__global__ void make_rows_kernel(const int32_t* last, const int32_t* draft, const int32_t* dlen, int B, int K,
                                 int32_t* tokens, int32_t* n_rows, unsigned long long* stamp) {
  next_may_launch();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B * (K + 1)) return;
  const int b = i / (K + 1), j = i % (K + 1);
  wait_for_earlier();
  const int32_t lt = last[b];
  const int m = lt < 0 ? 0 : min(max(dlen[b], 0), K);
  tokens[i] = lt < 0 ? -1 : (j == 0 ? lt : (j <= m ? draft[b * K + j - 1] : -1));
  if (j == 0) n_rows[b] = lt < 0 ? 0 : 1 + m;
  if (stamp && i == 0) *stamp = device_ns();
}

}  // namespace
}  // namespace laser

LASER_API laser_status laser_pool_free(laser_pool* pool) {
  if (!pool) return LASER_OK;
  int dev = 0;
  const bool other = cudaGetDevice(&dev) == cudaSuccess && dev != pool->device;
  if (other) cudaSetDevice(pool->device);
  cudaDeviceSynchronize();                 // lookups on any stream may still read it
  laser::pooled_free(pool->memory, nullptr);
  if (other) cudaSetDevice(dev);
  delete pool;
  return LASER_OK;
}

LASER_API laser_status laser_pool_build(const int32_t* tokens, int64_t n_tokens,
                                        const int64_t* group_offsets, int32_t n_groups,
                                        int32_t n_min, int32_t n_max, void* stream_,
                                        laser_pool** out) {
  using namespace laser;
  LASER_REQUIRE(tokens && group_offsets && out, "null argument");
  LASER_REQUIRE(n_tokens >= 1 && n_tokens < (int64_t(1) << 31), "n_tokens = %lld outside [1, 2^31)", (long long)n_tokens);
  LASER_REQUIRE(n_groups >= 1, "n_groups = %d", n_groups);
  LASER_REQUIRE(n_min >= 1 && n_min <= n_max && n_max <= kMaxN, "suffix range [%d, %d] outside [1, %d]", n_min, n_max, kMaxN);
  LASER_REQUIRE(group_offsets[0] == 0 && group_offsets[n_groups] == n_tokens, "group_offsets must span [0, n_tokens]");
  for (int g = 0; g < n_groups; ++g)
    LASER_REQUIRE(group_offsets[g] <= group_offsets[g + 1], "group_offsets not ascending at %d", g);
  cudaStream_t stream = as_stream(stream_);
  laser_pool* P = new laser_pool();
  P->n_tokens = n_tokens; P->n_groups = n_groups; P->n_min = n_min; P->n_max = n_max;
  struct Guard { laser_pool* p; ~Guard() { if (p) laser_pool_free(p); } } guard{P};

  LASER_CUDA(cudaGetDevice(&P->device));

  // Groups by size: what fits shared memory, in three classes of its use (one, two and three CTAs an SM), the larger first, and
  // the rest, which are sorted together: larger groups, and tiny ones where they are many.  The positions of the first come first
  // in the position arrays, those of the sorted groups behind.
  const size_t N = size_t(n_tokens);
  auto class_of = [&](int64_t size) { int c = 0; while (c < kClasses && size <= kClassMax[c]) ++c; return c; };   // 0: large
  int count[kClasses + 1] = {}, n_tiny = 0;
  int64_t sum[kClasses + 1] = {}, tiny_sum = 0;
  for (int g = 0; g < n_groups; ++g) {
    const int64_t size = group_offsets[g + 1] - group_offsets[g];
    const int c = class_of(size);
    ++count[c]; sum[c] += size;
    if (size < kTinyGroup) { ++n_tiny; tiny_sum += size; }
  }
  const int64_t least = n_tiny >= kManyTiny ? kTinyGroup : 0;    // of a group in shared memory
  if (least) { count[kClasses] -= n_tiny; sum[kClasses] -= tiny_sum; count[0] += n_tiny; sum[0] += tiny_sum; }
  // [n_groups] ids, [n_groups + 1] starts: of the groups in shared memory their runs' place, of the others their place among those
  // (none where all are sorted)
  const bool listed = count[0] < n_groups;
  std::unique_ptr<uint32_t[]> lists(listed ? new (std::nothrow) uint32_t[size_t(n_groups) * 2 + 1] : nullptr);
  if (listed && !lists) { set_error("no host memory for %d groups", n_groups); return LASER_ERR_OOM; }
  uint32_t *const h_id = lists.get(), *const h_at = h_id + n_groups;
  int fill[kClasses + 1];
  int64_t place[kClasses + 1];
  const int n_small_groups = n_groups - count[0];
  int64_t n_small = 0;
  for (int c = 1, f = 0; c <= kClasses; ++c) { fill[c] = f; place[c] = n_small; f += count[c]; n_small += sum[c]; }
  fill[0] = n_small_groups; place[0] = 0;
  for (int g = 0; listed && g < n_groups; ++g) {
    const int64_t size = group_offsets[g + 1] - group_offsets[g];
    const int c = size < least ? 0 : class_of(size);
    h_id[fill[c]] = uint32_t(g);
    h_at[fill[c]++] = uint32_t(place[c]);
    place[c] += size;
  }
  if (listed) h_at[n_groups] = uint32_t(sum[0]);
  const int64_t n_sorted = sum[0];
  const size_t M = size_t(n_sorted);

  // One allocation for the index, sized before any key is counted; one for the build's own buffers.
  const size_t slots = size_t(region_base(n_tokens, n_groups));
  LASER_REQUIRE(slots < kNoSlot, "%lld tokens in %d groups are too many for one index", (long long)n_tokens, n_groups);
  auto padded = [](size_t bytes) { return (bytes + 255) & ~size_t(255); };
  const size_t b_tok = padded(N * 4), b_goff = padded((size_t(n_groups) + 1) * 8), b_tab = padded(slots * 8), b_pos = padded((N + 32) * 4);
  P->device_bytes = int64_t(b_tok + b_goff + (n_max - n_min + 1) * (b_tab + b_pos));
  LASER_TRY(pooled_alloc(&P->memory, size_t(P->device_bytes), stream));
  uint8_t* at = static_cast<uint8_t*>(P->memory);
  auto take = [&](auto** p, size_t bytes) { *p = reinterpret_cast<std::remove_reference_t<decltype(*p)>>(at); at += bytes; };
  take(&P->tokens, b_tok);
  take(&P->group_offsets, b_goff);
  IndexLevels lvs{};
  for (int n = n_min; n <= n_max; ++n) {
    auto& lv = P->level[n];
    take(&lv.table, b_tab);
    take(&lv.positions, b_pos);
    lvs.table[n] = lv.table; lvs.positions[n] = lv.positions;
  }
  LASER_CUDA(cudaMemcpyAsync(P->tokens, tokens, N * 4, cudaMemcpyDefault, stream));
  LASER_CUDA(cudaMemcpyAsync(P->group_offsets, group_offsets, (size_t(n_groups) + 1) * 8, cudaMemcpyHostToDevice, stream));

  // The sorted groups' n-grams go through one sort for as many n as 32-bit slot numbers and 64 M pairs hold.
  const int levels = n_max - n_min + 1;
  const int batch = int(std::max<size_t>(1, std::min({size_t(levels), size_t(kNoSlot) / slots, (size_t(64) << 20) / std::max<size_t>(M, 1)})));
  int slot_bits = 1;             // all that kNoSlot needs to sort behind every slot
  while (slot_bits < 32 && (slots * batch) >> slot_bits) ++slot_bits;
  const size_t pairs = M * batch;
  size_t cub_bytes = 0;
  if (M) {
    cub::DoubleBuffer<uint32_t> kb(nullptr, nullptr), vb(nullptr, nullptr);
    LASER_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, cub_bytes, kb, vb, int64_t(pairs), 0, slot_bits, stream));
  }
  constexpr size_t kCounters = (2 * kMaxN + 3) * 8;   // distinct keys per n, the largest token, n-grams of the sorted groups per n
  const size_t b_lists = listed ? (size_t(n_groups) * 2 + 1) * 4 : 0;
  struct Tmp { void* p = nullptr; cudaStream_t s; ~Tmp() { pooled_free(p, s); } } tmp{nullptr, stream};
  LASER_TRY(pooled_alloc(&tmp.p, 4 * padded(pairs * 4) + padded(kCounters) + padded(b_lists) + cub_bytes + 256, stream));
  at = static_cast<uint8_t*>(tmp.p);
  uint32_t *slot_of, *slot_alt, *pos, *pos_alt;
  unsigned long long* counters;
  uint32_t* d_id;
  uint8_t* cub_tmp;
  take(&slot_of, padded(pairs * 4)); take(&slot_alt, padded(pairs * 4)); take(&pos, padded(pairs * 4)); take(&pos_alt, padded(pairs * 4));
  take(&counters, padded(kCounters)); take(&d_id, padded(b_lists)); take(&cub_tmp, cub_bytes);
  const uint32_t* d_at = d_id + n_groups;
  int* max_tok = reinterpret_cast<int*>(counters + kMaxN + 1);
  unsigned long long* n_valid = counters + kMaxN + 2;
  if (listed) LASER_CUDA(cudaMemcpyAsync(d_id, lists.get(), b_lists, cudaMemcpyHostToDevice, stream));
  LASER_CUDA(cudaMemsetAsync(counters, 0, kCounters, stream));
  LASER_CUDA(cudaMemsetAsync(max_tok, 0xff, 4, stream));
  for (int n = n_min; n <= n_max; ++n) LASER_CUDA(cudaMemsetAsync(P->level[n].positions + N, 0xff, 32 * 4, stream));
  if (least)                     // (so many regions are cleared as whole tables)
    for (int n = n_min; n <= n_max; ++n) LASER_CUDA(cudaMemsetAsync(P->level[n].table, 0xff, slots * 8, stream));
  size_t done = 0;
  for (int c = 1; c <= kClasses; ++c) {
    if (!count[c]) continue;
    auto index = [&](auto kernel, unsigned threads) -> laser_status {
      const size_t smem = group_smem(kClassMax[c - 1]);
      LASER_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)));
      LASER_CUDA(launch_overlapped(kernel, dim3(unsigned(count[c]), unsigned(n_max - n_min + 1)), threads, smem, stream, P->tokens,
                                   P->group_offsets, d_id + done, d_at + done, done == 0 ? 1 : 0, n_min, lvs, counters, max_tok));
      return LASER_OK;
    };
    LASER_TRY(c == 1 ? index(index_group_kernel<1024, 1>, 1024) : c == 2 ? index(index_group_kernel<512, 2>, 512) : index(index_group_kernel<512, 3>, 512));
    count_launch();
    done += size_t(count[c]);
  }
  if (M) {
    const SortedGroups lg{listed ? d_id + done : nullptr, listed ? d_at + done : nullptr, count[0]};
    const unsigned blocks = unsigned(ceil_div<size_t>(M, kInsertBlock));
    for (int l0 = 0; l0 < lg.n && !least; l0 += 65535)
      clear_regions_kernel<<<dim3(16, unsigned(std::min(lg.n - l0, 65535)), unsigned(levels)), kKeyThreads, 0, stream>>>(
          lvs, n_min, P->group_offsets, lg, l0);
    count_launch();
    for (int n0 = n_min; n0 <= n_max; n0 += batch) {
      const int nb = std::min(batch, n_max - n0 + 1);
      const int64_t count = int64_t(M) * nb;
      insert_sorted_kernel<<<dim3(blocks, unsigned(nb)), kKeyThreads, 0, stream>>>(P->tokens, P->group_offsets, lg, n_sorted, n0, lvs,
                                                                                  uint32_t(slots), slot_of, pos, n_valid, max_tok);
      cub::DoubleBuffer<uint32_t> kb(slot_of, slot_alt), vb(pos, pos_alt);
      LASER_CUDA(cub::DeviceRadixSort::SortPairs(cub_tmp, cub_bytes, kb, vb, count, 0, slot_bits, stream));
      index_runs_kernel<<<unsigned(ceil_div<int64_t>(count, kKeyThreads)), kKeyThreads, 0, stream>>>(
          kb.Current(), vb.Current(), count, n_small, n0, lvs, uint32_t(slots), n_valid, counters);
      count_launch(2);
      LASER_CUDA(cudaGetLastError());
    }
  }
  unsigned long long h_cnt[kMaxN + 2] = {};
  LASER_CUDA(cudaMemcpyAsync(h_cnt, counters, sizeof(h_cnt), cudaMemcpyDeviceToHost, stream));
  LASER_CUDA(cudaStreamSynchronize(stream));
  for (int n = n_min; n <= n_max; ++n) P->level[n].n_keys = int64_t(h_cnt[n]);
  P->vocab_bound = int32_t(uint32_t(h_cnt[kMaxN + 1])) + 1;
  guard.p = nullptr;
  *out = P;
  return LASER_OK;
}

LASER_API laser_status laser_pool_info(const laser_pool* pool, int64_t* n_tokens, int64_t* n_keys,
                                       int64_t* device_bytes) {
  using namespace laser;
  LASER_REQUIRE(pool, "null pool");
  if (n_tokens) *n_tokens = pool->n_tokens;
  if (n_keys) { *n_keys = 0; for (int n = pool->n_min; n <= pool->n_max; ++n) *n_keys += pool->level[n].n_keys; }
  if (device_bytes) *device_bytes = pool->device_bytes;
  return LASER_OK;
}

LASER_API laser_status laser_draft(const laser_pool* pool, const int32_t* tails, const int32_t* tail_len,
                                   const int32_t* group_id, int32_t B, const laser_params* p,
                                   int32_t* draft, int32_t* draft_len, int32_t* match_n, void* stream_) {
  using namespace laser;
  LASER_REQUIRE(pool && tails && tail_len && group_id && p && draft && draft_len && match_n, "null argument");
  LASER_REQUIRE(B >= 0, "B = %d", B);
  LASER_REQUIRE(p->K >= 1 && p->K <= kMaxK, "K = %d outside [1, %d]", p->K, kMaxK);
  LASER_REQUIRE(p->n_min >= pool->n_min && p->n_max <= pool->n_max && p->n_min <= p->n_max,
                "suffix range [%d, %d] outside the pool's [%d, %d]", p->n_min, p->n_max, pool->n_min, pool->n_max);
  LASER_REQUIRE(p->max_occ >= 0 && p->min_draft >= 0, "max_occ / min_draft negative");
  if (B == 0) return LASER_OK;
  cudaStream_t stream = as_stream(stream_);
  const PoolView pv = view_of(pool);
  const bool big = (p->max_occ == 0 || p->max_occ > 64);
  const size_t hist = size_t(pool->vocab_bound) * sizeof(uint32_t);
  if (big && hist > kHistMost) {
    set_error("vocabulary bound %d too large for the unlimited-occurrence path", pool->vocab_bound);
    return LASER_ERR_UNSUPPORTED;
  }
  void* scratch = nullptr;
  if (big) LASER_TRY(scratch_get(SCRATCH_DRAFT, sizeof(int32_t) * (size_t(WORK_HEAD) + 3 * size_t(B)), &scratch));
  DraftArgs a{tails, tail_len, group_id, B, p->K, p->n_min, p->n_max, p->min_draft, p->max_occ,
              draft, draft_len, match_n, static_cast<int32_t*>(scratch), pool->n_tokens};
  LASER_CUDA(launch_overlapped(draft_warp_kernel, dim3(unsigned(ceil_div(B, kDraftWarps))), kDraftWarps * 32, 0, stream, pv, a));
  count_launch();
  if (big) {
    const size_t smem = std::max(hist + kBigList * sizeof(uint32_t), p->max_occ > 0 && p->max_occ <= kBigList ? kTeamSmem : kBigSmem);
    const uint32_t list_cap = uint32_t((smem - hist) / sizeof(uint32_t));
    // (the same for all launches: another thread's may come between this and the next line)
    LASER_CUDA(cudaFuncSetAttribute(draft_cta_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kHistMost + kBigList * sizeof(uint32_t))));
    LASER_CUDA(launch_overlapped(draft_cta_kernel, dim3(unsigned(std::min(B, 148))), kBigThreads, smem, stream, pv, a, pool->vocab_bound, list_cap));
    count_launch();
  }
  LASER_CUDA(cudaGetLastError());
  return LASER_OK;
}

LASER_API laser_status laser_draft_temp(const laser_pool* pool, const int32_t* tails, const int32_t* tail_len,
                                        const int32_t* group_id, const int32_t* hist, const int32_t* hist_len,
                                        int64_t hist_stride, int32_t B, const laser_params* p,
                                        int32_t* draft, int32_t* draft_len, int32_t* match_n, void* stream_) {
  using namespace laser;
  LASER_REQUIRE(pool && tails && tail_len && group_id && hist && hist_len && p && draft && draft_len && match_n, "null argument");
  LASER_REQUIRE(B >= 0 && hist_stride >= 0, "B = %d, hist_stride = %lld", B, (long long)hist_stride);
  LASER_REQUIRE(p->K >= 1 && p->K <= kMaxK, "K = %d outside [1, %d]", p->K, kMaxK);
  LASER_REQUIRE(p->n_min >= pool->n_min && p->n_max <= pool->n_max && p->n_min <= p->n_max,
                "suffix range [%d, %d] outside the pool's [%d, %d]", p->n_min, p->n_max, pool->n_min, pool->n_max);
  LASER_REQUIRE(p->max_occ >= 1 && p->max_occ <= 64 && p->min_draft >= 0,
                "max_occ = %d: the temporary-branch draft keeps 1..64 occurrences", p->max_occ);
  if (B == 0) return LASER_OK;
  cudaStream_t stream = as_stream(stream_);
  const PoolView pv = view_of(pool);
  DraftArgs a{tails, tail_len, group_id, B, p->K, p->n_min, p->n_max, p->min_draft, p->max_occ,
              draft, draft_len, match_n, nullptr, pool->n_tokens};
  TempArgs t{hist, hist_len, hist_stride};
  LASER_CUDA(launch_overlapped(draft_temp_kernel, dim3(unsigned(ceil_div(B, kDraftWarps))), kDraftWarps * 32, 0, stream, pv, a, t));
  count_launch();
  LASER_CUDA(cudaGetLastError());
  return LASER_OK;
}

LASER_API laser_status laser_draft_tree(const laser_pool* pool, const int32_t* tails, const int32_t* tail_len,
                                        const int32_t* group_id, const int32_t* hist, const int32_t* hist_len,
                                        int64_t hist_stride, int32_t B, const laser_params* p, int32_t* draft,
                                        int32_t* draft_parents, int32_t* draft_len, int32_t* match_n, void* stream_) {
  using namespace laser;
  LASER_REQUIRE(pool && tails && tail_len && group_id && p && draft && draft_parents && draft_len && match_n, "null argument");
  LASER_REQUIRE((hist == nullptr) == (hist_len == nullptr), "hist and hist_len come together");
  LASER_REQUIRE(B >= 0 && hist_stride >= 0, "B = %d, hist_stride = %lld", B, (long long)hist_stride);
  LASER_REQUIRE(p->K >= 1 && p->K <= kTreeK, "K = %d outside [1, %d]", p->K, kTreeK);
  LASER_REQUIRE(p->n_min >= pool->n_min && p->n_max <= pool->n_max && p->n_min <= p->n_max,
                "suffix range [%d, %d] outside the pool's [%d, %d]", p->n_min, p->n_max, pool->n_min, pool->n_max);
  LASER_REQUIRE(p->max_occ >= 1 && p->max_occ <= 64 && p->min_draft >= 0,
                "max_occ = %d: tree drafting keeps 1..64 occurrences", p->max_occ);
  if (B == 0) return LASER_OK;
  const PoolView pv = view_of(pool);
  DraftArgs a{tails, tail_len, group_id, B, p->K, p->n_min, p->n_max, p->min_draft, p->max_occ,
              draft, draft_len, match_n, nullptr, pool->n_tokens};
  TempArgs t{hist, hist_len, hist_stride};
  LASER_CUDA(launch_overlapped(draft_tree_kernel, dim3(unsigned(B)), 32, 0, as_stream(stream_), pv, a, t, draft_parents));
  count_launch();
  LASER_CUDA(cudaGetLastError());
  return LASER_OK;
}

namespace laser {
laser_status make_rows(const int32_t* last_token, const int32_t* draft, const int32_t* draft_len, int32_t B, int32_t K, int32_t* tokens,
                       int32_t* n_rows, unsigned long long* stamp, cudaStream_t stream) {
  LASER_REQUIRE(last_token && draft && draft_len && tokens && n_rows, "null argument");
  LASER_REQUIRE(B >= 0 && K >= 0, "B = %d, K = %d", B, K);
  if (B == 0) return LASER_OK;
  LASER_CUDA(launch_overlapped(make_rows_kernel, dim3(unsigned(ceil_div(B * (K + 1), 256))), 256, 0, stream, last_token, draft, draft_len,
                               B, K, tokens, n_rows, stamp));
  count_launch();
  return LASER_OK;
}

laser_status make_rows_tree(const int32_t* last_token, const int32_t* draft, const int32_t* draft_parents, const int32_t* draft_len,
                            int32_t B, int32_t K, int32_t* tokens, int32_t* parents, int32_t* n_rows, unsigned long long* stamp,
                            cudaStream_t stream) {
  LASER_REQUIRE(last_token && draft && draft_parents && draft_len && tokens && parents && n_rows, "null argument");
  LASER_REQUIRE(B >= 0 && K >= 0, "B = %d, K = %d", B, K);
  if (B == 0) return LASER_OK;
  LASER_CUDA(launch_overlapped(make_tree_rows_kernel, dim3(unsigned(ceil_div(B * (K + 1), 256))), 256, 0, stream, last_token, draft,
                               draft_parents, draft_len, B, K, tokens, parents, n_rows, stamp));
  count_launch();
  return LASER_OK;
}
}  // namespace laser

LASER_API laser_status laser_make_rows_tree(const int32_t* last_token, const int32_t* draft, const int32_t* draft_parents,
                                            const int32_t* draft_len, int32_t B, int32_t K, int32_t* tokens,
                                            int32_t* parents, int32_t* n_rows, void* stream) {
  return laser::make_rows_tree(last_token, draft, draft_parents, draft_len, B, K, tokens, parents, n_rows, nullptr, laser::as_stream(stream));
}

LASER_API laser_status laser_make_rows(const int32_t* last_token, const int32_t* draft,
                                       const int32_t* draft_len, int32_t B, int32_t K,
                                       int32_t* tokens, int32_t* n_rows, void* stream) {
  return laser::make_rows(last_token, draft, draft_len, B, K, tokens, n_rows, nullptr, laser::as_stream(stream));
}
