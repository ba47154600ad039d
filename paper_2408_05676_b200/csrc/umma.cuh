// tcgen05 (fifth-generation tensor core) instruction wrappers: shared-memory matrix descriptors,
// the bf16 MMA into a tensor-memory accumulator, commits onto mbarriers and tensor-memory loads.
#pragma once
#include <stdint.h>

namespace laser {

// Shared-memory matrix descriptor: K-major tile, 128-byte swizzle, rows 128 B apart, groups
// of 8 rows 1024 B apart.
__device__ __forceinline__ uint64_t umma_desc(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= uint64_t((smem_addr & 0x3FFFF) >> 4);        // start address
  d |= uint64_t(1024 >> 4) << 32;                   // stride byte offset between 8-row groups
  d |= uint64_t(1) << 46;                           // descriptor version of this architecture
  d |= uint64_t(2) << 61;                           // 128-byte swizzle
  return d;
}
// The loops that issue copies and MMAs run on a whole warp, with one elected lane doing the issuing: these instructions take
// their operands from uniform registers, and in a loop that only one lane runs every operand is first moved there (60
// cycles an MMA against about 15).  7B verify step, 64 cached tokens, 4 layers: 9 rows 409 -> 397 us, 36 rows 469 -> 443, 144
// rows 530 -> 522; precise mode, which issues twice the MMAs per weight block: 9 rows 499 -> 426, 144 rows 788 -> 745.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t e;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(e));
  return e;
}
__device__ __forceinline__ void umma_commit(uint32_t bar, uint32_t elected) {
  asm volatile("{\n.reg .pred q;\nsetp.ne.b32 q, %1, 0;\n@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}"
               ::"r"(bar), "r"(elected) : "memory");
}
// One K block: 64 elements = four K steps of 32 bytes inside the swizzle span.
__device__ __forceinline__ void umma_kblock(uint32_t tmem_d, uint64_t wdesc, uint64_t adesc, uint32_t idesc, uint32_t accumulate, uint32_t elected) {
  asm volatile(
      "{\n.reg .pred p, q;\n.reg .b64 w1, w2, w3, a1, a2, a3;\nsetp.ne.b32 q, %5, 0;\nsetp.ne.b32 p, %4, 0;\n"
      "add.s64 w1, %1, 2;\nadd.s64 a1, %2, 2;\nadd.s64 w2, %1, 4;\nadd.s64 a2, %2, 4;\nadd.s64 w3, %1, 6;\nadd.s64 a3, %2, 6;\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], w1, a1, %3, 1;\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], w2, a2, %3, 1;\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], w3, a3, %3, 1;\n}"
      ::"r"(tmem_d), "l"(wdesc), "l"(adesc), "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}
// The same in a CTA pair (cluster ranks 0 and 1): one 256-row MMA over both, each CTA holding half of both operands in its
// shared memory; issued by rank 0.
__device__ __forceinline__ void umma_kblock_pair(uint32_t tmem_d, uint64_t wdesc, uint64_t adesc, uint32_t idesc, uint32_t accumulate, uint32_t elected) {
  asm volatile(
      "{\n.reg .pred p, q;\n.reg .b64 w1, w2, w3, a1, a2, a3;\nsetp.ne.b32 q, %5, 0;\nsetp.ne.b32 p, %4, 0;\n"
      "add.s64 w1, %1, 2;\nadd.s64 a1, %2, 2;\nadd.s64 w2, %1, 4;\nadd.s64 a2, %2, 4;\nadd.s64 w3, %1, 6;\nadd.s64 a3, %2, 6;\n"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], w1, a1, %3, 1;\n"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], w2, a2, %3, 1;\n"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], w3, a3, %3, 1;\n}"
      ::"r"(tmem_d), "l"(wdesc), "l"(adesc), "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}
// arrives on the barrier at the same shared-memory offset in every CTA named by the rank mask
__device__ __forceinline__ void umma_commit_pair(uint32_t bar, uint32_t rank_mask, uint32_t elected) {
  asm volatile(
      "{\n.reg .pred q;\n.reg .b16 m;\ncvt.u16.u32 m, %1;\nsetp.ne.b32 q, %2, 0;\n"
      "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], m;\n}"
      ::"r"(bar), "r"(rank_mask), "r"(elected) : "memory");
}
// 16 consecutive fp32 columns of this thread's TMEM lane (no wait: pair with tmem_ld_wait)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

}  // namespace laser
