// Inline-PTX building blocks of the tensor-core kernels (sm_100a): mbarriers, bulk-tensor copies, TMEM
// management and loads, tcgen05 MMA issue for int8 operands, shared-memory descriptors.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace adaption {
namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// The same test, but the hardware may keep the thread suspended for up to `hint_ns` while the phase
// is incomplete (it resumes as soon as the phase completes): far fewer polling instructions.
__device__ __forceinline__ bool mbar_try_wait_suspend(uint32_t bar, uint32_t parity, uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}
// True in exactly one lane of a converged warp.  Code guarded by it still has its operands computed
// warp-uniformly outside the guard, which lets the compiler keep them in uniform registers (the
// tensor-core and bulk-copy instructions take uniform-register operands).
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile(
      "{\n"
      ".reg .pred P;\n"
      "elect.sync _|P, 0xffffffff;\n"
      "selp.u32 %0, 1, 0, P;\n"
      "}\n"
      : "=r"(pred));
  return pred != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// PAIR: the copy lands in this CTA's shared memory but reports its bytes to an mbarrier that may
// live in the other CTA of the pair (the leader's "full" barrier).
template <bool PAIR>
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x,
                                            int y) {
  if (PAIR)
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
        "l"(map), "r"(bar), "r"(x), "r"(y)
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
        "l"(map), "r"(bar), "r"(x), "r"(y)
        : "memory");
}
template <bool PAIR>
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z) {
  if (PAIR)
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
        "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z)
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
        "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z)
        : "memory");
}
template <bool PAIR>
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z,
                                            int w) {
  if (PAIR)
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
        "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z), "r"(w)
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
        "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z), "r"(w)
        : "memory");
}
template <bool PAIR>
__device__ __forceinline__ void tma_load_im2col(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c,
                                                int w, int h, int n, uint16_t off_w, uint16_t off_h) {
  if (PAIR)
    asm volatile(
        "cp.async.bulk.tensor.4d.im2col.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};" ::"r"(dst),
        "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"(off_w), "h"(off_h)
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};" ::"r"(dst),
        "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"(off_w), "h"(off_h)
        : "memory");
}
template <bool PAIR>
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
  if (PAIR)
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
                 "r"(ncols)
                 : "memory");
  else
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
                 "r"(ncols)
                 : "memory");
}
template <bool PAIR>
__device__ __forceinline__ void tmem_relinquish() {
  if (PAIR)
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  else
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
template <bool PAIR>
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  if (PAIR)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
  else
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
}
// ---- CTA-pair plumbing
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of the same shared-memory offset in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t mapa_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// generic-proxy writes to shared memory become visible to bulk copies
__device__ __forceinline__ void fence_async_shared() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// Arrive on `bar` once every MMA issued so far by this thread has retired.  PAIR: the arrival is
// delivered to the barrier at the same offset in both CTAs of the pair.
template <bool PAIR>
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  if (PAIR)
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            bar),
        "h"((uint16_t)3)
        : "memory");
  else
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}
// Operand descriptors are passed as 32-bit halves: the high word (group stride, version, swizzle)
// is the same for every operand tile of a launch, the low word is the shared-memory address in
// 16-byte units, so stepping along K or to another plane is one 32-bit add.
// PAIR: one instruction computes a 256-row tile across the two CTAs of the pair: each CTA supplies
// its own 128 rows of A and half of the B rows, and receives its 128 rows of the result in its TMEM.
template <bool PAIR>
__device__ __forceinline__ void mma_i8(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi,
                                       uint32_t idesc, uint32_t accumulate, uint32_t b_desc_hi) {
  if (PAIR)
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        ".reg .b64 da, db;\n"
        "setp.ne.b32 p, %5, 0;\n"
        "mov.b64 da, {%1, %3};\n"
        "mov.b64 db, {%2, %6};\n"
        "tcgen05.mma.cta_group::2.kind::i8 [%0], da, db, %4, p;\n"
        "}\n" ::"r"(d_tmem),
        "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate), "r"(b_desc_hi)
        : "memory");
  else
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        ".reg .b64 da, db;\n"
        "setp.ne.b32 p, %5, 0;\n"
        "mov.b64 da, {%1, %3};\n"
        "mov.b64 db, {%2, %6};\n"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %4, p;\n"
        "}\n" ::"r"(d_tmem),
        "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate), "r"(b_desc_hi)
        : "memory");
}
template <bool PAIR>
__device__ __forceinline__ void mma_i8(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                       uint32_t accumulate) {
  mma_i8<PAIR>(d_tmem, a_lo, b_lo, desc_hi, idesc, accumulate, desc_hi);
}
// eight consecutive columns
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, int32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
// sixteen consecutive columns: the first eight into `lo`, the next eight into `hi`
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, int32_t (&lo)[8], int32_t (&hi)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(lo[0]), "=r"(lo[1]), "=r"(lo[2]), "=r"(lo[3]), "=r"(lo[4]), "=r"(lo[5]), "=r"(lo[6]), "=r"(lo[7]),
        "=r"(hi[0]), "=r"(hi[1]), "=r"(hi[2]), "=r"(hi[3]), "=r"(hi[4]), "=r"(hi[5]), "=r"(hi[6]), "=r"(hi[7])
      : "r"(taddr)
      : "memory");
}
// thirty-two consecutive columns in one instruction (a TMEM load costs about the same latency
// whatever its width, so the widest form that the register budget allows drains fastest)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, int32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
// two runs of sixteen columns, `step` columns apart
__device__ __forceinline__ void tmem_ld16x2(uint32_t taddr, uint32_t step, int32_t (&r)[32]) {
#pragma unroll
  for (int h = 0; h < 2; ++h)
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[16 * h + 0]), "=r"(r[16 * h + 1]), "=r"(r[16 * h + 2]), "=r"(r[16 * h + 3]), "=r"(r[16 * h + 4]),
          "=r"(r[16 * h + 5]), "=r"(r[16 * h + 6]), "=r"(r[16 * h + 7]), "=r"(r[16 * h + 8]), "=r"(r[16 * h + 9]),
          "=r"(r[16 * h + 10]), "=r"(r[16 * h + 11]), "=r"(r[16 * h + 12]), "=r"(r[16 * h + 13]),
          "=r"(r[16 * h + 14]), "=r"(r[16 * h + 15])
        : "r"(taddr + (h ? step : 0u))
        : "memory");
}
__device__ __forceinline__ void pin_after_wait32(int32_t (&r)[32]) {
  asm volatile(""
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                 "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                 "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}
// Placed after tcgen05.wait::ld: ties the loaded registers to that point so that no use of them can
// be scheduled before the wait (the load fills them asynchronously).
__device__ __forceinline__ void pin_after_wait(int32_t (&r)[8]) {
  asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile whose rows are BK bytes long and
// swizzled with a span of BK bytes: eight-row groups are `sbo` bytes apart; the two 16-byte
// halves of one 32-byte k-step are adjacent (leading offset 1).
// High word: group stride / 16 in bits 0-13, descriptor version 1 in bit 14, swizzle in bits 29-31.
__device__ __forceinline__ uint32_t smem_desc_hi(uint32_t sbo, uint32_t layout_type) {
  return ((sbo >> 4) & 0x3FFFu) | (1u << 14) | (layout_type << 29);
}
// Low word: start address / 16 in bits 0-13, leading offset 1 in bits 16-29.
__device__ __forceinline__ uint32_t smem_desc_lo(uint32_t saddr) {
  return ((saddr >> 4) & 0x3FFFu) | (1u << 16);
}


// One 32-byte k-step of a tile, issued as a single instruction sequence so that the issuing thread
// spends as few instructions per MMA as possible (its instruction stream, not the tensor pipe, is
// what limits the mainloop otherwise).  Operand descriptors: low words a0/a1/b0/b1, high word dhi
// for A and dhb for B.  acc = 0 overwrites the accumulators (first k-step of a tile).
#define ADAPTION_MMA_KSTEP_2X2(CG)                                                              \
  asm volatile(                                                                                 \
      "{\n"                                                                                     \
      ".reg .pred p, q;\n"                                                                      \
      ".reg .b64 da0, da1, db0, db1;\n"                                                         \
      "setp.ne.b32 p, %12, 0;\n"                                                                \
      "setp.eq.b32 q, %7, %7;\n"                                                                \
      "mov.b64 da0, {%3, %7};\n"                                                                \
      "mov.b64 da1, {%4, %7};\n"                                                                \
      "mov.b64 db0, {%5, %13};\n"                                                               \
      "mov.b64 db1, {%6, %13};\n"                                                               \
      "tcgen05.mma.cta_group::" CG ".kind::i8 [%0], da0, db0, %8, p;\n"                         \
      "tcgen05.mma.cta_group::" CG ".kind::i8 [%1], da0, db1, %9, p;\n"                         \
      "tcgen05.mma.cta_group::" CG ".kind::i8 [%1], da1, db0, %10, q;\n"                        \
      "tcgen05.mma.cta_group::" CG ".kind::i8 [%2], da1, db1, %11, p;\n"                        \
      "}\n" ::"r"(d0),                                                                          \
      "r"(d1), "r"(d2), "r"(a0), "r"(a1), "r"(b0), "r"(b1), "r"(dhi), "r"(id_ss), "r"(id_su),  \
      "r"(id_us), "r"(id_uu), "r"(acc), "r"(dhb)                                                \
      : "memory")

template <bool PAIR>
__device__ __forceinline__ void mma_kstep_2x2(uint32_t d0, uint32_t d1, uint32_t d2, uint32_t a0, uint32_t a1,
                                              uint32_t b0, uint32_t b1, uint32_t dhi, uint32_t id_ss,
                                              uint32_t id_su, uint32_t id_us, uint32_t id_uu, uint32_t acc,
                                              uint32_t dhb) {
  // hi*hi -> d0 (weight 2^16); hi*lo and lo*hi -> d1 (weight 2^8); lo*lo -> d2 (weight 1)
  if (PAIR)
    ADAPTION_MMA_KSTEP_2X2("2");
  else
    ADAPTION_MMA_KSTEP_2X2("1");
}
#undef ADAPTION_MMA_KSTEP_2X2

template <int NAX, int NBW, bool PAIR>
__device__ __forceinline__ void mma_kstep(uint32_t d0, uint32_t d1, uint32_t d2, uint32_t a0, uint32_t a1,
                                          uint32_t b0, uint32_t b1, uint32_t dhi, uint32_t id_ss, uint32_t id_su,
                                          uint32_t id_us, uint32_t id_uu, uint32_t acc, uint32_t dhb) {
  if (NAX == 2 && NBW == 2) {
    mma_kstep_2x2<PAIR>(d0, d1, d2, a0, a1, b0, b1, dhi, id_ss, id_su, id_us, id_uu, acc, dhb);
  } else if (NAX == 2 && NBW == 1) {
    mma_i8<PAIR>(d0, a0, b0, dhi, id_ss, acc, dhb);          // hi*w    weight 2^8
    mma_i8<PAIR>(d1, a1, b0, dhi, id_us, acc, dhb);          // lo*w    weight 1
  } else if (NAX == 1 && NBW == 2) {
    mma_i8<PAIR>(d0, a0, b0, dhi, id_ss, acc, dhb);          // x*hi    weight 2^8
    mma_i8<PAIR>(d1, a0, b1, dhi, id_su, acc, dhb);          // x*lo    weight 1
  } else {
    mma_i8<PAIR>(d0, a0, b0, dhi, id_ss, acc, dhb);
  }
}

template <int NAX, int NBW, bool PAIR>
__device__ __forceinline__ void mma_kstep(uint32_t d0, uint32_t d1, uint32_t d2, uint32_t a0, uint32_t a1,
                                          uint32_t b0, uint32_t b1, uint32_t dhi, uint32_t id_ss, uint32_t id_su,
                                          uint32_t id_us, uint32_t id_uu, uint32_t acc) {
  mma_kstep<NAX, NBW, PAIR>(d0, d1, d2, a0, a1, b0, b1, dhi, id_ss, id_su, id_us, id_uu, acc, dhi);
}

// `STEPS` consecutive k-steps of one product, as one instruction sequence.
#define ADAPTION_MMA_STEPS(CG, MORE)                                       \
  asm volatile(                                                             \
      "{\n"                                                                 \
      ".reg .pred p, q;\n"                                                  \
      ".reg .b32 x, y;\n"                                                   \
      ".reg .b64 da, db;\n"                                                 \
      "setp.ne.b32 p, %5, 0;\n"                                             \
      "setp.eq.b32 q, %3, %3;\n"                                            \
      "mov.b64 da, {%1, %3};\n"                                             \
      "mov.b64 db, {%2, %3};\n"                                             \
      "tcgen05.mma.cta_group::" CG ".kind::i8 [%0], da, db, %4, p;\n" MORE "}\n" ::"r"(d), \
      "r"(a), "r"(b), "r"(dhi), "r"(id), "r"(acc)                            \
      : "memory")
#define ADAPTION_MMA_NEXT(CG, OFF)                                          \
  "add.u32 x, %1, " OFF ";\n"                                               \
  "add.u32 y, %2, " OFF ";\n"                                               \
  "mov.b64 da, {x, %3};\n"                                                  \
  "mov.b64 db, {y, %3};\n"                                                  \
  "tcgen05.mma.cta_group::" CG ".kind::i8 [%0], da, db, %4, q;\n"
template <bool PAIR>
__device__ __forceinline__ void mma_single_kblock(uint32_t d, uint32_t a, uint32_t b, uint32_t dhi, uint32_t id,
                                                  int ksteps, uint32_t acc) {
  if (PAIR) {
    if (ksteps == 4)
      ADAPTION_MMA_STEPS("2", ADAPTION_MMA_NEXT("2", "2") ADAPTION_MMA_NEXT("2", "4") ADAPTION_MMA_NEXT("2", "6"));
    else if (ksteps == 3)
      ADAPTION_MMA_STEPS("2", ADAPTION_MMA_NEXT("2", "2") ADAPTION_MMA_NEXT("2", "4"));
    else if (ksteps == 2)
      ADAPTION_MMA_STEPS("2", ADAPTION_MMA_NEXT("2", "2"));
    else
      ADAPTION_MMA_STEPS("2", "");
  } else {
    if (ksteps == 4)
      ADAPTION_MMA_STEPS("1", ADAPTION_MMA_NEXT("1", "2") ADAPTION_MMA_NEXT("1", "4") ADAPTION_MMA_NEXT("1", "6"));
    else if (ksteps == 3)
      ADAPTION_MMA_STEPS("1", ADAPTION_MMA_NEXT("1", "2") ADAPTION_MMA_NEXT("1", "4"));
    else if (ksteps == 2)
      ADAPTION_MMA_STEPS("1", ADAPTION_MMA_NEXT("1", "2"));
    else
      ADAPTION_MMA_STEPS("1", "");
  }
}
#undef ADAPTION_MMA_STEPS
#undef ADAPTION_MMA_NEXT

// All k-steps of one k-block (1, 2 or 4 of them; with PARTIAL also 3).  a0: low descriptor word of the first
// plane of A, b0 of B; the other planes and the k-steps are fixed offsets in 16-byte units.
template <int NAX, int NBW, bool PAIR, bool PARTIAL>
__device__ __forceinline__ void mma_kblock(uint32_t d0, uint32_t d1, uint32_t d2, uint32_t a0, uint32_t off_a1, uint32_t b0,
                                           uint32_t b_u, uint32_t dhi, uint32_t id_ss, uint32_t id_su, uint32_t id_us,
                                           uint32_t id_uu, int ksteps, uint32_t acc) {
  if (NAX == 1 && NBW == 1) {
    mma_single_kblock<PAIR>(d0, a0, b0, dhi, id_ss, ksteps, acc);
    return;
  }
  const uint32_t a1 = a0 + off_a1, b1 = b0 + b_u;
  mma_kstep<NAX, NBW, PAIR>(d0, d1, d2, a0, a1, b0, b1, dhi, id_ss, id_su, id_us, id_uu, acc);
  if (ksteps > 1) mma_kstep<NAX, NBW, PAIR>(d0, d1, d2, a0 + 2u, a1 + 2u, b0 + 2u, b1 + 2u, dhi, id_ss, id_su, id_us, id_uu, 1u);
  if (ksteps > 2) {
    mma_kstep<NAX, NBW, PAIR>(d0, d1, d2, a0 + 4u, a1 + 4u, b0 + 4u, b1 + 4u, dhi, id_ss, id_su, id_us, id_uu, 1u);
    if (!PARTIAL || ksteps > 3)
      mma_kstep<NAX, NBW, PAIR>(d0, d1, d2, a0 + 6u, a1 + 6u, b0 + 6u, b1 + 6u, dhi, id_ss, id_su, id_us, id_uu, 1u);
  }
}

// The same in warp-uniform control flow: every lane of the issuing warp comes along and the one with `issue` != 0 (elect_one
// once, before the loop) issues.  Operands stay in uniform registers that way, and a rolled loop stays in the instruction
// cache of a scheduler that also runs the epilogue: as straight-line code in a branch of one lane, filter taps copied once
// (two 8-bit instructions each) took 270 to 320 cycles apiece, twice what the tensor core needs.
template <bool PAIR>
__device__ __forceinline__ void mma_i8_if(uint32_t issue, uint32_t d, uint32_t a, uint32_t b, uint32_t dha, uint32_t dhb,
                                          uint32_t id, uint32_t acc) {
#define ADAPTION_MMA_IF(CG)                                              \
  asm volatile(                                                          \
      "{\n"                                                              \
      ".reg .pred p, e;\n"                                               \
      ".reg .b64 da, db;\n"                                              \
      "setp.ne.b32 e, %0, 0;\n"                                          \
      "setp.ne.b32 p, %7, 0;\n"                                          \
      "mov.b64 da, {%2, %4};\n"                                          \
      "mov.b64 db, {%3, %5};\n"                                          \
      "@e tcgen05.mma.cta_group::" CG ".kind::i8 [%1], da, db, %6, p;\n" \
      "}\n" ::"r"(issue),                                                \
      "r"(d), "r"(a), "r"(b), "r"(dha), "r"(dhb), "r"(id), "r"(acc)      \
      : "memory")
  if (PAIR)
    ADAPTION_MMA_IF("2");
  else
    ADAPTION_MMA_IF("1");
#undef ADAPTION_MMA_IF
}
// One 32-byte k-step of all products.
template <int NAX, int NBW, bool PAIR>
__device__ __forceinline__ void mma_kstep_if(uint32_t issue, uint32_t d0, uint32_t d1, uint32_t d2, uint32_t a0, uint32_t a1,
                                             uint32_t b0, uint32_t b1, uint32_t dha, uint32_t dhb, uint32_t id_ss,
                                             uint32_t id_su, uint32_t id_us, uint32_t id_uu, uint32_t acc) {
  mma_i8_if<PAIR>(issue, d0, a0, b0, dha, dhb, id_ss, acc);
  if (NAX == 2 && NBW == 2) {
    mma_i8_if<PAIR>(issue, d1, a0, b1, dha, dhb, id_su, acc);
    mma_i8_if<PAIR>(issue, d2, a1, b1, dha, dhb, id_uu, acc);
    mma_i8_if<PAIR>(issue, d1, a1, b0, dha, dhb, id_us, 1u);
  } else if (NAX == 2) {
    mma_i8_if<PAIR>(issue, d1, a1, b0, dha, dhb, id_us, acc);
  } else if (NBW == 2) {
    mma_i8_if<PAIR>(issue, d1, a0, b1, dha, dhb, id_su, acc);
  }
}
template <int NAX, int NBW, bool PAIR>
__device__ __forceinline__ void mma_kblock_if(uint32_t issue, uint32_t d0, uint32_t d1, uint32_t d2, uint32_t a0, uint32_t off_a1,
                                              uint32_t b0, uint32_t b_u, uint32_t dha, uint32_t dhb, uint32_t id_ss,
                                              uint32_t id_su, uint32_t id_us, uint32_t id_uu, int ksteps, uint32_t acc) {
#pragma unroll 1
  for (int k = 0; k < ksteps; ++k) {
    mma_kstep_if<NAX, NBW, PAIR>(issue, d0, d1, d2, a0, a0 + off_a1, b0, b0 + b_u, dha, dhb, id_ss, id_su, id_us, id_uu, acc);
    acc = 1u;
    a0 += 2u;
    b0 += 2u;
  }
}
template <bool PAIR>
__device__ __forceinline__ void tc_commit_if(uint32_t issue, uint32_t bar) {
  if (PAIR)
    asm volatile(
        "{\n"
        ".reg .pred e;\n"
        "setp.ne.b32 e, %2, 0;\n"
        "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n"
        "}\n" ::"r"(bar),
        "h"((uint16_t)3), "r"(issue)
        : "memory");
  else
    asm volatile(
        "{\n"
        ".reg .pred e;\n"
        "setp.ne.b32 e, %1, 0;\n"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
        "}\n" ::"r"(bar),
        "r"(issue)
        : "memory");
}

// Instruction descriptor: int32 accumulate, 8-bit operands with independent signedness,
// both K-major, M = 128, N = bn.
__device__ __forceinline__ uint32_t make_idesc(bool a_signed, bool b_signed, int bn, int m) {
  return (2u << 4) | ((a_signed ? 1u : 0u) << 7) | ((b_signed ? 1u : 0u) << 10) |
         ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

}  // namespace
}  // namespace adaption
