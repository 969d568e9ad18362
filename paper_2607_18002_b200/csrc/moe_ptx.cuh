// Inline-PTX wrappers for the sm_100a features the persistent kernels use: mbarriers, tiled TMA loads,
// tcgen05 (UMMA) issue / commit / TMEM loads, proxy fences and scoped loads and stores.
#pragma once
#include <cuda.h>
#include <stdint.h>

namespace moe {

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(void* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(void* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try(void* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// orders what this thread wrote or saw before what it writes after, for all of the device
__device__ __forceinline__ void fence_acq_rel_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
// L2 policy of bytes that nobody reads a second time
__device__ __forceinline__ unsigned long long l2_evict_first() {
  unsigned long long p;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ unsigned long long l2_evict_normal() {
  unsigned long long p;
  asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_commit(void* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tc_mma_bf16(unsigned d_tmem, unsigned long long adesc,
                                            unsigned long long bdesc, unsigned idesc,
                                            unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_ld32(unsigned taddr, unsigned (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
// 16 TMEM lanes x 32 columns in the fragment layout of an m16n8 accumulator: for column group j (8 columns) thread i
// holds row i / 4, columns 8 j + 2 (i % 4) and + 1 in r[4 j], r[4 j + 1], and the same columns of row i / 4 + 8 in r[4 j + 2],
// r[4 j + 3]
__device__ __forceinline__ void tc_ld_frag(unsigned taddr, unsigned (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// 16 lanes x 64 columns: register pair (4 j + 2 r, + 1) is row lane / 4 + 8 r, columns 8 j + 2 (lane % 4) and the next
__device__ __forceinline__ void tc_ld_frag64(unsigned taddr, unsigned (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
// 16 TMEM lanes x 16 columns: thread i holds column 4 j + i % 4 of row i / 4 in r[2 j] and of row i / 4 + 8 in r[2 j + 1] (twice
// the rate of the layout above)
__device__ __forceinline__ void tc_ld_pairs(unsigned taddr, unsigned (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x128b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr)
      : "memory");
}
// four 8x8 matrices of 16-bit elements, stored transposed: thread i gives the address of a 16-byte row of matrix i / 8
__device__ __forceinline__ void st_matrix4_trans(unsigned saddr, unsigned r0, unsigned r1, unsigned r2, unsigned r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared::cta.b16 [%0], {%1, %2, %3, %4};" ::"r"(saddr), "r"(r0), "r"(r1), "r"(r2), "r"(r3)
               : "memory");
}
__device__ __forceinline__ void tc_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}
__device__ __forceinline__ void cp_async_4(unsigned dst_smem, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst_smem), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_16(unsigned dst_smem, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst_smem), "l"(src) : "memory");
}
// the mbarrier receives one arrival when all cp.async issued so far by this thread have landed
__device__ __forceinline__ void cp_async_arrive_noinc(void* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}
__device__ __forceinline__ void fence_async_proxy_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_async_proxy() {
  asm volatile("fence.proxy.async;" ::: "memory");
}
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned ld_acquire_sys(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_sys(unsigned* p, unsigned v) {
  asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// a word in shared memory
__device__ __forceinline__ unsigned ld_acquire_cta(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_cta(unsigned* p, unsigned v) {
  asm volatile("st.release.cta.shared.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_volatile(const int* p) {
  return *reinterpret_cast<const volatile int*>(p);
}

// UMMA shared-memory descriptor of a K-major operand whose rows are row_bytes (64 or 128)
// wide and swizzled with the matching pattern; 8-row groups lie 8 * row_bytes apart.
__device__ __forceinline__ unsigned long long umma_desc(unsigned saddr, unsigned row_bytes) {
  unsigned long long d = (unsigned long long)((saddr & 0x3ffffu) >> 4);
  d |= 1ull << 16;                                   // leading byte offset (unused for swizzled K-major)
  d |= (unsigned long long)((8u * row_bytes) >> 4) << 32;   // stride byte offset between 8-row groups
  d |= 1ull << 46;                                   // descriptor version (sm_100)
  d |= (row_bytes == 128u ? 2ull : 4ull) << 61;      // SWIZZLE_128B : SWIZZLE_64B
  return d;
}
// instruction descriptor: D fp32, A/B bf16, both K-major, M = 128, N = 256
constexpr unsigned kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((256u >> 3) << 17) | ((128u >> 4) << 24);



// ------------------------------------------------------------------ CTA pairs (cluster of two)
__device__ __forceinline__ unsigned cluster_ctarank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {      // every thread of both CTAs
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared::cluster address of the same shared-memory object in CTA `rank` of the cluster
__device__ __forceinline__ unsigned map_to_cta(const void* p, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(unsigned cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// behind a fence of the caller's that orders what the arrival hands over
__device__ __forceinline__ void mbar_arrive_relaxed(unsigned cluster_addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// A stage's rows are in place in the shared memory of the CTA that says so, where the pair's MMAs read them: written by cp.async of this
// CTA's threads, seen complete by the caller and fenced for the tensor core, so the release is to this CTA.  (To the cluster, once a
// k-block, it takes longer than the k-block: one token 56 -> 129 us a pass, 777 tokens 1120 -> 2604.)
__device__ __forceinline__ void mbar_arrive_remote(unsigned cluster_addr) {
  asm volatile("mbarrier.arrive.release.cta.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// wait that synchronises with arrivals made by the other CTA of the pair
__device__ __forceinline__ bool mbar_try_cluster(void* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// wait for relaxed arrivals of the other CTA: a fence of the caller's orders what follows
__device__ __forceinline__ bool mbar_try_relaxed(void* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void st_cluster_v4(unsigned cluster_addr, uint4 v) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// one lane of a converged warp.  The compiler knows a branch on elect.sync for a region of one thread: instructions that take uniform
// registers (TMA, MMA, commit) are then issued as they stand
__device__ __forceinline__ bool elect_one() {
  unsigned e;
  asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 r;\n\telect.sync r|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0;
}
// arrives on the barrier at the same shared-memory offset in both CTAs once this thread's MMAs of the pair so far retire
__device__ __forceinline__ void tc_commit_pair(void* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(smem_u32(bar)),
               "h"((unsigned short)3)
               : "memory");
}

// The weights of one k-block by one CTA of a pair, by one thread: expect_tx (of the rows' bytes too) on the leader's stage barrier, the
// stand-in arrivals (tiles without a gather), the go-ahead for those that bring the rows, and the box of 128 weight rows with its L2
// policy.  The next stage's barrier is tested first and the result read last, as with the MMAs: returns whether that stage is free.
__device__ __forceinline__ bool pair_issue_kblock(unsigned bar, unsigned tx, unsigned standin_bar, unsigned standin_n, unsigned go_bar,
                                                  unsigned has_go, unsigned sW, const CUtensorMap* tmw, int x, int wblk, int expert,
                                                  unsigned long long w_policy, unsigned next_empty_bar, unsigned next_parity) {
  unsigned ready;
  asm volatile(
      "{\n\t.reg .pred pgo, pst, pn;\n\t.reg .b32 z;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 pn, [%13], %14;\n\t"
      "setp.ne.b32 pst, %4, 0;\n\t"
      "setp.ne.b32 pgo, %6, 0;\n\t"
      "mov.b32 z, 0;\n\t"
      "mbarrier.arrive.expect_tx.shared::cluster.b64 _, [%1], %2;\n\t"
      "@pgo mbarrier.arrive.shared::cta.b64 _, [%5];\n\t"
      "@pst mbarrier.arrive.shared::cta.b64 _, [%3], %4;\n\t"
      "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%7], [%8, {%9, z, z, %10, %11}], [%1], %12;\n\t"
      "selp.u32 %0, 1, 0, pn;\n\t}"
      : "=r"(ready)
      : "r"(bar), "r"(tx), "r"(standin_bar), "r"(standin_n), "r"(go_bar), "r"(has_go), "r"(sW),
        "l"(reinterpret_cast<unsigned long long>(tmw)), "r"(x), "r"(wblk), "r"(expert), "l"(w_policy), "r"(next_empty_bar), "r"(next_parity)
      : "memory");
  return ready != 0;
}

// ... the weights of a second k-block in the same stage
__device__ __forceinline__ void pair_issue_weights(unsigned bar, unsigned sW, const CUtensorMap* tmw, int x, int wblk, int expert,
                                                   unsigned long long w_policy) {
  asm volatile(
      "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%1], [%2, {%3, %6, %6, %4, %5}], [%0], %7;"
      ::"r"(bar), "r"(sW), "l"(reinterpret_cast<unsigned long long>(tmw)), "r"(x), "r"(wblk), "r"(expert), "r"(0), "l"(w_policy)
      : "memory");
}

// The activation boxes of one k-block by one CTA of a pair, by one thread: up to three, a_rows rows apart
__device__ __forceinline__ void pair_issue_rows(unsigned bar, int x, unsigned sX, const CUtensorMap* tma, int ay, unsigned a_boxes,
                                                unsigned a_rows) {
  asm volatile(
      "{\n\t.reg .pred pa1, pa2, pa3;\n\t.reg .b32 st, sA1, ay1, sA2, ay2;\n\t"
      "setp.ge.u32 pa1, %5, 1;\n\t"
      "setp.ge.u32 pa2, %5, 2;\n\t"
      "setp.ge.u32 pa3, %5, 3;\n\t"
      "shl.b32 st, %6, 7;\n\t"
      "add.u32 sA1, %2, st;\n\t"
      "add.s32 ay1, %4, %6;\n\t"
      "add.u32 sA2, sA1, st;\n\t"
      "add.s32 ay2, ay1, %6;\n\t"
      "@pa1 cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%2], [%3, {%1, %4}], [%0];\n\t"
      "@pa2 cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [sA1], [%3, {%1, ay1}], [%0];\n\t"
      "@pa3 cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [sA2], [%3, {%1, ay2}], [%0];\n\t}"
      ::"r"(bar), "r"(x), "r"(sX), "l"(reinterpret_cast<unsigned long long>(tma)), "r"(ay), "r"(a_boxes), "r"(a_rows)
      : "memory");
}

// The four MMAs of one tile's k-block, where another tile's follow against the same rows
__device__ __forceinline__ void pair_mma_half(unsigned d_tmem, unsigned long long adesc, unsigned long long bdesc, unsigned idesc,
                                              unsigned accumulate_first) {
  asm volatile(
      "{\n\t.reg .pred p0, p1;\n\t.reg .b64 a1, a2, a3, b1, b2, b3;\n\t"
      "setp.ne.b32 p0, %4, 0;\n\t"
      "setp.eq.b32 p1, 0, 0;\n\t"
      "add.u64 a1, %1, 2;\n\tadd.u64 a2, %1, 4;\n\tadd.u64 a3, %1, 6;\n\t"
      "add.u64 b1, %2, 2;\n\tadd.u64 b2, %2, 4;\n\tadd.u64 b3, %2, 6;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], a1, b1, %3, p1;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], a2, b2, %3, p1;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], a3, b3, %3, p1;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate_first)
      : "memory");
}

// One k-block of the pair's MMAs, by one thread: the next stage's barrier is tested first and
// the result is only read after the four MMAs and the commit have been issued, so that the barrier's
// shared-memory round trip hides behind the issue of the MMAs.  Returns whether the next stage is already full.
__device__ __forceinline__ bool pair_mma_kblock(unsigned d_tmem, unsigned long long adesc, unsigned long long bdesc,
                                                unsigned idesc, unsigned accumulate_first, unsigned empty_bar,
                                                unsigned next_full_bar, unsigned next_parity) {
  unsigned ready;
  asm volatile(
      "{\n\t.reg .pred p0, p1, pn;\n\t.reg .b16 m;\n\t.reg .b64 a1, a2, a3, b1, b2, b3;\n\t"
      "mov.b16 m, 3;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 pn, [%7], %8;\n\t"
      "setp.ne.b32 p0, %5, 0;\n\t"
      "setp.eq.b32 p1, 0, 0;\n\t"
      "add.u64 a1, %2, 2;\n\tadd.u64 a2, %2, 4;\n\tadd.u64 a3, %2, 6;\n\t"
      "add.u64 b1, %3, 2;\n\tadd.u64 b2, %3, 4;\n\tadd.u64 b3, %3, 6;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%1], %2, %3, %4, p0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%1], a1, b1, %4, p1;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%1], a2, b2, %4, p1;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%1], a3, b3, %4, p1;\n\t"
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%6], m;\n\t"
      "selp.u32 %0, 1, 0, pn;\n\t}"
      : "=r"(ready)
      : "r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate_first), "r"(empty_bar),
        "r"(next_full_bar), "r"(next_parity)
      : "memory");
  return ready != 0;
}
// two fp32 lanes per instruction, each rounded like the scalar operation
__device__ __forceinline__ unsigned long long f32x2(float lo, float hi) {
  unsigned long long v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
  return v;
}
__device__ __forceinline__ float2 f32x2_parts(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ unsigned long long mul_f32x2(unsigned long long a, unsigned long long b) {
  unsigned long long v;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}
__device__ __forceinline__ unsigned long long fma_f32x2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long v;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
  return v;
}
// One e4m3 k-block of a small tile, by one thread: both halves of the weight tile as M = 128 operands against the same few token rows, into
// the columns from d and from d + half on; the commit that frees the stage and (end_of_group) the one that hands the group of partials over.
// Returns whether the next stage is already full (tested first, read last, as in pair_mma_kblock).
__device__ __forceinline__ bool f8_small_kblock(unsigned d_tmem, unsigned long long w0desc, unsigned long long w1desc,
                                                unsigned long long xdesc, unsigned idesc, unsigned half, unsigned pfull_bar, unsigned end_of_group,
                                                unsigned empty_bar, unsigned next_full_bar, unsigned next_parity) {
  unsigned ready;
  asm volatile(
      "{\n\t.reg .pred p0, p1, pg, pn;\n\t.reg .b32 d1;\n\t.reg .b64 x1, x2, x3, a1, a2, a3, b1, b2, b3;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 pn, [%10], %11;\n\t"
      "setp.ne.b32 p0, 0, 0;\n\t"
      "setp.eq.b32 p1, 0, 0;\n\t"
      "setp.ne.b32 pg, %7, 0;\n\t"
      "add.u32 d1, %1, %9;\n\t"
      "add.u64 x1, %4, 2;\n\tadd.u64 x2, %4, 4;\n\tadd.u64 x3, %4, 6;\n\t"
      "add.u64 a1, %2, 2;\n\tadd.u64 a2, %2, 4;\n\tadd.u64 a3, %2, 6;\n\t"
      "add.u64 b1, %3, 2;\n\tadd.u64 b2, %3, 4;\n\tadd.u64 b3, %3, 6;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%1], %2, %4, %5, p0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%1], a1, x1, %5, p1;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%1], a2, x2, %5, p1;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%1], a3, x3, %5, p1;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [d1], %3, %4, %5, p0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [d1], b1, x1, %5, p1;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [d1], b2, x2, %5, p1;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [d1], b3, x3, %5, p1;\n\t"
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%8];\n\t"
      "@pg tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%6];\n\t"
      "selp.u32 %0, 1, 0, pn;\n\t}"
      : "=r"(ready)
      : "r"(d_tmem), "l"(w0desc), "l"(w1desc), "l"(xdesc), "r"(idesc), "r"(pfull_bar), "r"(end_of_group), "r"(empty_bar), "r"(half),
        "r"(next_full_bar), "r"(next_parity)
      : "memory");
  return ready != 0;
}
// One e4m3 k-block (128 elements = four 32-element MMAs) into a fresh partial buffer, by one thread, then the two commits (partial full, stage
// empty).  The barriers of the next k-block, its stage and its partial buffer, are tested first and the results read last.
__device__ __forceinline__ void f8_mma_kblock(unsigned d_tmem, unsigned long long adesc, unsigned long long bdesc,
                                              unsigned idesc, unsigned pfull_bar, unsigned empty_bar, unsigned next_full_bar, unsigned next_parity,
                                              unsigned next_pempty_bar, unsigned next_pparity, bool& ready, bool& drained) {
  unsigned r, d;
  asm volatile(
      "{\n\t.reg .pred p0, p1, pn, pp;\n\t.reg .b64 a1, a2, a3, b1, b2, b3;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 pn, [%8], %9;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 pp, [%10], %11;\n\t"
      "setp.ne.b32 p0, 0, 0;\n\t"
      "setp.eq.b32 p1, 0, 0;\n\t"
      "add.u64 a1, %3, 2;\n\tadd.u64 a2, %3, 4;\n\tadd.u64 a3, %3, 6;\n\t"
      "add.u64 b1, %4, 2;\n\tadd.u64 b2, %4, 4;\n\tadd.u64 b3, %4, 6;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%2], %3, %4, %5, p0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%2], a1, b1, %5, p1;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%2], a2, b2, %5, p1;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%2], a3, b3, %5, p1;\n\t"
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%6];\n\t"
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%7];\n\t"
      "selp.u32 %0, 1, 0, pn;\n\t"
      "selp.u32 %1, 1, 0, pp;\n\t}"
      : "=r"(r), "=r"(d)
      : "r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(pfull_bar), "r"(empty_bar), "r"(next_full_bar), "r"(next_parity),
        "r"(next_pempty_bar), "r"(next_pparity)
      : "memory");
  ready = r != 0;
  drained = d != 0;
}
// The weights of one k-block of the single-CTA kernel, by one thread: expect_tx (of the rows' bytes too), the stand-in arrivals (tiles whose
// rows one thread loads), the go-ahead for those that bring the rows, and the box of 256 weight rows with its L2 policy.  Returns whether
// the next stage is already free.
__device__ __forceinline__ bool single_issue_kblock(unsigned bar, unsigned tx, unsigned standin_n, unsigned go_bar, unsigned sW,
                                                    const CUtensorMap* tmw, int x, int c1, int c2, int c3, int c4, unsigned long long w_policy,
                                                    unsigned next_empty_bar, unsigned next_parity) {
  unsigned ready;
  asm volatile(
      "{\n\t.reg .pred pst, pn;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 pn, [%13], %14;\n\t"
      "setp.ne.b32 pst, %3, 0;\n\t"
      "mbarrier.arrive.expect_tx.shared::cta.b64 _, [%1], %2;\n\t"
      "mbarrier.arrive.shared::cta.b64 _, [%4];\n\t"
      "@pst mbarrier.arrive.shared::cta.b64 _, [%1], %3;\n\t"
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%5], [%6, {%7, %8, %9, %10, %11}], [%1], %12;\n\t"
      "selp.u32 %0, 1, 0, pn;\n\t}"
      : "=r"(ready)
      : "r"(bar), "r"(tx), "r"(standin_n), "r"(go_bar), "r"(sW), "l"(reinterpret_cast<unsigned long long>(tmw)), "r"(x), "r"(c1), "r"(c2),
        "r"(c3), "r"(c4), "l"(w_policy), "r"(next_empty_bar), "r"(next_parity)
      : "memory");
  return ready != 0;
}
// The activation rows of a k-block, by one thread: a box, and behind it a second one of 32 rows
__device__ __forceinline__ void single_issue_rows(unsigned bar, int x, unsigned sA, const CUtensorMap* tma, int ay, unsigned a_boxes) {
  asm volatile(
      "{\n\t.reg .pred pa2;\n\t.reg .b32 sA1, ay1;\n\t"
      "setp.ge.u32 pa2, %5, 2;\n\t"
      "add.u32 sA1, %2, 4096;\n\t"
      "add.s32 ay1, %4, 32;\n\t"
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%2], [%3, {%1, %4}], [%0];\n\t"
      "@pa2 cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [sA1], [%3, {%1, ay1}], [%0];\n\t}"
      ::"r"(bar), "r"(x), "r"(sA), "l"(reinterpret_cast<unsigned long long>(tma)), "r"(ay), "r"(a_boxes)
      : "memory");
}
}  // namespace moe
