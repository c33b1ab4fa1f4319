// What the tensor-core convolution kernels share: PTX wrappers (mbarriers, TMA, tcgen05), the shared-memory operand
// descriptor, the 32-bit forms of Eq. 4 and the residual rescale of Section 3.3, and the tensor-map encoders.
// Every translation unit gets its own copy (internal linkage).
#pragma once

#include <cuda.h>
#include <climits>

#include "hq_internal.cuh"

namespace {

constexpr int kTileC = 128;                   // output channels per tile = MMA M = TMEM lanes
constexpr unsigned long long kWaitBudgetNs = 2000000000ull;   // 2 s per wait
constexpr uint32_t kSuspendNs = 1000000;      // longest single suspension of a waiting thread (it looks at the abort flag in between)

// ---------------------------------------------------------------- PTX wrappers ---------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// The same, with leave for the hardware to keep the thread suspended for up to `ns` while the phase is not complete.
__device__ __forceinline__ bool mbar_try_wait_for(uint32_t bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(ns) : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait.  Returns false when the budget ran out or another role already aborted.
template <class Ctl>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, Ctl* ctl, uint32_t* status, uint32_t code,
                                          unsigned long long budget_ns = kWaitBudgetNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (true) {
    if (mbar_try_wait_for(bar, parity, kSuspendNs)) return true;
    if (ctl->abort_flag) return false;
    if (global_ns() - t0 > budget_ns) {
      ctl->abort_flag = 1;
      atomicCAS(status, 0u, code);
      return false;
    }
  }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y) : "memory");
}
// The same copy with an L2 eviction priority.  Activations and residual tiles that a layer reads exactly once per
// channel tile are fetched "evict first": they then make room before the output lines the layer is writing, and the
// next layer (which starts at the end this one wrote last, see TcParams::rev) finds more of its input in the L2.
__device__ __forceinline__ unsigned long long policy_evict_first() {
  unsigned long long pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void tma_load_2d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y,
                                                 unsigned long long pol) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "l"(pol) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void tma_load_im2col(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                                int c, int w, int h, int n, uint16_t off_w, uint16_t off_h) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"(off_w), "h"(off_h) : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c, int w, int h, int n) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n) : "memory");
}
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, uint32_t src, int c, int w, int h, int n) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
               ::"l"(map), "r"(src), "r"(c), "r"(w), "r"(h), "r"(n) : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(map), "r"(src), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
template <int EPI_THREADS>
__device__ __forceinline__ uint32_t epi_bar_and(uint32_t v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred p, 1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r) : "r"(v), "n"(EPI_THREADS) : "memory");
  return r;
}

// True in exactly one lane of a converged warp; tells the compiler the guarded region is
// single-lane, which lets it keep TMA / MMA operands in uniform registers.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(pred));
  return pred != 0;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void mma_i8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// ---- two-CTA forms (cta_group::2).  `in_cta(addr, r)` names the same shared-memory offset in the cluster's CTA r.
__device__ __forceinline__ uint32_t in_cta(uint32_t addr, uint32_t cta_rank) {
  uint32_t r; asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(cta_rank)); return r;
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_alloc2(uint32_t dst_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void mma_i8_2cta(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
// arrives on ONE barrier (of either CTA of the pair) when the pair's MMAs issued so far have completed
__device__ __forceinline__ void mma_commit_2cta(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// loads of a CTA pair: the bytes land in the issuing CTA's shared memory and are counted on the leading CTA's barrier
__device__ __forceinline__ void tma_load_2d_2cta(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(in_cta(bar, 0)), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_load_im2col_2cta(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                                     int c, int w, int h, int n, uint16_t off_w, uint16_t off_h) {
  asm volatile(
      "cp.async.bulk.tensor.4d.im2col.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
      ::"r"(dst), "l"(map), "r"(in_cta(bar, 0)), "r"(c), "r"(w), "r"(h), "r"(n), "h"(off_w), "h"(off_h) : "memory");
}
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, int (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld8_issue(uint32_t taddr, int (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(taddr) : "memory");
}
// Keeps what is computed from the loaded registers below the wait: used above it, they could also be given to something else
// while the load is still going to write them.
template <int N>
__device__ __forceinline__ void tie(int (&v)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) asm volatile("" : "+r"(v[i]));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// 16 lanes x 32 columns in the layout of an MMA accumulator fragment: thread T (t4 = T / 4, q2 = T % 4) receives, for
// every group g of eight columns, v[4g + 0/1] = lane t4, columns 8g + 2 q2 + 0/1 and v[4g + 2/3] = lane t4 + 8, same columns.
__device__ __forceinline__ void tmem_ld_frag16(uint32_t taddr, int (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr) : "memory");
}
// Four 8 x 8 matrices of 16-bit elements, transposed on the way: register g of thread T (t4, q2 as above) holds the elements
// (t4, 2 q2) and (t4, 2 q2 + 1) of matrix g, whose column n is the 16 contiguous bytes at the address thread 8 g + n supplies.
// With the weight rows in the order of encode_paired_rows_map an element is two neighbouring channels of one pixel.
__device__ __forceinline__ void stmatrix_t_x4(uint32_t row_addr, unsigned r0, unsigned r1, unsigned r2, unsigned r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};"
               ::"r"(row_addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3) : "memory");
}
__device__ __forceinline__ void ldmatrix_t_x4(uint32_t row_addr, unsigned (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(row_addr) : "memory");
}
// four values -> four bytes (s0 lowest), clamped to the unsigned / signed 8-bit range by two chained saturating packs
template <bool OSIGNED>
__device__ __forceinline__ unsigned sat_pack4(int s0, int s1, int s2, int s3) {
  unsigned w23, w;
  if (OSIGNED) {
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(w23) : "r"(s3), "r"(s2), "r"(0));
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(w) : "r"(s1), "r"(s0), "r"(w23));
  } else {
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(w23) : "r"(s3), "r"(s2), "r"(0));
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(w) : "r"(s1), "r"(s0), "r"(w23));
  }
  return w;
}
// Saturating conversion to a byte.  The packing form of the convert (second source -> byte 0) is a single
// integer-pipe instruction; the plain cvt.sat.u8.s32 measured at twice its issue cost.
__device__ __forceinline__ int sat_u8(int x) {
  int d; asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %1;" : "=r"(d) : "r"(0), "r"(x)); return d;
}
__device__ __forceinline__ int sat_s8(int x) {
  int d; asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %1;" : "=r"(d) : "r"(0), "r"(x)); return d;
}

// 4 x 4 bytes turned round inside each quad of lanes: lane i's word holds bytes (i, 0..3); afterwards (0..3, i).
__device__ __forceinline__ unsigned quad_transpose(unsigned w, int lane) {
  unsigned o = __shfl_xor_sync(0xffffffffu, w, 1);
  w = (lane & 1) ? __byte_perm(w, o, 0x3715) : __byte_perm(w, o, 0x6240);
  o = __shfl_xor_sync(0xffffffffu, w, 2);
  return (lane & 2) ? __byte_perm(w, o, 0x3276) : __byte_perm(w, o, 0x5410);
}

// Shared-memory matrix descriptor for a K-major operand tile whose rows are `bkb` bytes wide and
// stored with the matching TMA swizzle (32/64/128 B): 8-row groups are bkb*8 bytes apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t bkb) {
  const uint64_t layout = (bkb == 128) ? 2ull : (bkb == 64) ? 4ull : 6ull;
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);            // start address
  d |= (uint64_t)1 << 16;                            // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(((bkb * 8) >> 4) & 0x3FFF) << 32;  // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;                            // descriptor version for this architecture
  d |= layout << 61;
  return d;
}

// Per-thread (= per output channel) constants of the epilogue.
struct ChanConst {
  int b, sh;            // main branch multiplier; shift (c, or c - min(c,32) on the fast path)
  int sh1;              // fast path: min(c, 32), the part of the shift taken by the funnel shift
  int cmin31;           // fast path: min(c, 31)
  int pre;              // pre-shift form (SMALL == 2): 32 - min(c, 32), the accumulator is shifted left by it first
  long long r0;         // bias*b + 2^(c-1)
  int rb, rh, rsh;      // residual multiplier; fast path: rh = 2^(rc-9), rsh = rc-8; else rsh = rc
  long long rr0;        // general path: 2^(rc-1)
  int bias;
};

// One output value on the 32-bit fast path (Eq. 4; Section 3.3):
//   main      y  = hi32(acc*b + bias*b + 2^(c-1)) >> (c-32)                         (needs c >= 32)
//   residual  y += (hi32((r << 24) * rb) + 2^(rc-9)) >> (rc-8)                      (needs 9 <= rc)
// The residual form is exact: (r<<24)*rb >> 32 = floor(r*rb / 2^8), the rounding constant 2^(rc-1) is
// a multiple of 2^8, and the dropped low 8 bits of r*rb cannot carry across a multiple of 2^(rc-8).
// (A 64-bit multiply-add followed by a funnel shift measured no faster.)  `r` is the stored 8-bit
// residual, already extended.  SMALL: 1 when some channel of the warp has c < 32 (exact funnel-shift form with a
// saturation guard); 2 when, besides, every such channel's accumulator and bias are known to stay below 2^(c-2)
// (TcParams::acc_bits, checked per channel when the constants are set up): the accumulator is then shifted left by
// 32 - c first and r0 was shifted with it, (acc << pre) * b + (r0 << pre) = (acc * b + r0) << pre exactly and without
// overflow, and the plain form applies again at the cost of one shift.
// RN: every channel of the warp has a narrow residual pair (m, a, s) with (r*m + a) >> s equal to the residual
// term for all 256 values of r (found and checked exhaustively by residual_narrow_kernel); rb / rh / rsh hold
// m / a / s then, and a 32-bit multiply-add replaces the shift, multiply-high and add.
template <bool RES, bool RSIGNED, int SMALL, bool RN = false>
__device__ __forceinline__ int requant_fast(int acc, int r, const ChanConst& k) {
  if (SMALL == 2) acc <<= k.pre;
  const long long t1 = hq_mad_wide(acc, k.b, k.r0);
  int s;
  if (SMALL != 1) {
    s = (int)(t1 >> 32) >> k.sh;                       // c >= 32 (or pre-shifted): |s| < 2^30
  } else {
    // some channel of this warp has c < 32: take bits [c, c+32) of the 64-bit value with a funnel shift
    // and saturate to +-2^30 when the exact value does not fit (it is far outside every clamp range then,
    // and |residual term| < 2^30 keeps the sum inside INT32)
    const int hi = (int)(t1 >> 32);
    const unsigned lo = (unsigned)t1;
    const int s0 = (int)__funnelshift_rc(lo, (unsigned)hi, k.sh1);
    const int above = hi >> k.cmin31;                  // the bits above the window (sign for c >= 32)
    s = (above == (s0 >> 31)) ? (s0 >> k.sh) : (hi < 0 ? INT_MIN : INT_MAX);
    s = max(min(s, 1 << 30), -(1 << 30));
  }
  if (RES && RN) {
    s += (r * k.rb + k.rh) >> k.rsh;
  } else if (RES) {
    const unsigned top = (unsigned)r << 24;
    if (RSIGNED) s += (__mulhi((int)top, k.rb) + k.rh) >> k.rsh;
    else s += (int)((__umulhi(top, (unsigned)k.rb) + (unsigned)k.rh) >> k.rsh);
  }
  return s;
}

// Per-channel constants of one output channel (Eq. 4 and the residual rescale of Section 3.3), as the loops below want
// them: `fast` selects the 32-bit forms (see requant_fast), `pre` its pre-shift form.
template <class Params>
__device__ __forceinline__ ChanConst chan_const(const Params& p, int ch, bool fast, bool pre = false) {
  ChanConst k{};
  const bool live = ch < p.C;
  k.bias = (live && p.bias) ? p.bias[ch] : 0;
  k.b = live ? p.b[ch] : 0;
  const int cc = live ? p.c[ch] : 32;
  k.sh = cc;
  k.r0 = (long long)k.bias * (long long)k.b + (1LL << (cc - 1));
  if (p.res) {
    const int rcc = live ? p.rc[ch] : 32;
    k.rb = live ? p.rb[ch] : 0;
    k.rsh = rcc;
    k.rr0 = 1LL << (rcc - 1);
  }
  if (fast) {
    k.sh1 = k.sh < 32 ? k.sh : 32;
    k.cmin31 = k.sh < 31 ? k.sh : 31;
    k.sh -= k.sh1;
    k.pre = 32 - k.sh1;
    if (pre) k.r0 <<= k.pre;                                         // the pre-shift form (the caller checked its bounds)
    if (p.res) {
      if (k.rsh >= 40) { k.rb = 0; k.rh = 0; k.rsh = 1; }            // |r*rb| < 2^39: rounds to 0
      else { k.rh = 1 << (k.rsh - 9); k.rsh -= 8; }
    }
  }
  return k;
}

// ---------------------------------------------------------------- host side ------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
typedef CUresult (*EncodeIm2colFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const int*, const int*, cuuint32_t, cuuint32_t,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn g_encode_tiled = nullptr;
EncodeIm2colFn g_encode_im2col = nullptr;

bool load_driver_entry_points() {
  if (g_encode_tiled && g_encode_im2col) return true;
  cudaDriverEntryPointQueryResult qr;
  void* fn = nullptr;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qr) != cudaSuccess ||
      qr != cudaDriverEntryPointSuccess || !fn)
    return false;
  g_encode_tiled = (EncodeTiledFn)fn;
  fn = nullptr;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeIm2col", &fn, cudaEnableDefault, &qr) != cudaSuccess ||
      qr != cudaDriverEntryPointSuccess || !fn)
    return false;
  g_encode_im2col = (EncodeIm2colFn)fn;
  return true;
}

CUtensorMapSwizzle swizzle_for(int row_bytes) {
  return row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
       : row_bytes == 32 ? CU_TENSOR_MAP_SWIZZLE_32B : CU_TENSOR_MAP_SWIZZLE_NONE;
}

// 2-D byte map over a dense [rows][row_bytes] tensor with a box of `ib` bytes x `box_rows` rows.
bool encode_rows_map(CUtensorMap* map, const void* base, long long rows, long long row_bytes, int ib, int box_rows,
                     CUtensorMapSwizzle swz) {
  const cuuint64_t dims[2] = {(cuuint64_t)row_bytes, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)row_bytes};
  const cuuint32_t box[2] = {(cuuint32_t)ib, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return g_encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Weight rows in the order the fragment epilogue wants them on the accumulator lanes: of every sixteen output channels the
// eight even ones first, then the eight odd ones, so that a thread's two lanes (t4, t4 + 8) hold neighbouring channels.  A
// four-dimensional map walks them in that order: (K bytes, channel pairs, parity, sixteens).  `rows` is a multiple of 16; box:
// `ib` bytes of 128 rows.
bool encode_paired_rows_map(CUtensorMap* map, const void* base, long long rows, long long row_bytes, int ib, CUtensorMapSwizzle swz) {
  const cuuint64_t dims[4] = {(cuuint64_t)row_bytes, 8, 2, (cuuint64_t)(rows / 16)};
  const cuuint64_t strides[3] = {(cuuint64_t)(2 * row_bytes), (cuuint64_t)row_bytes, (cuuint64_t)(16 * row_bytes)};
  const cuuint32_t box[4] = {(cuuint32_t)ib, 8, 2, kTileC / 16};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return g_encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// im2col-mode map over the NHWC activations of a convolution, `bkb` channels x `pixels` output pixels per copy: (C, W, H, N)
// with byte strides; base pixels range over [-pad, W + pad - (kw-1)) so that the hardware's pixel walk equals the output
// raster.  A tensor below the mode's minimum that has ConvArgs::in_slack is declared with more images than it holds (what
// lies in them only reaches pixels past the last one).
bool encode_im2col_map(CUtensorMap* map, const ConvArgs& a, int bkb, int pixels) {
  const long long image = a.pitch_n ? a.pitch_n : (long long)a.cin * a.w * a.h;
  long long images = a.n;
  if (a.in_slack && images * image < kIm2colMinTensorBytes) images = (kIm2colMinTensorBytes + image - 1) / image;
  const cuuint64_t dims[4] = {(cuuint64_t)a.cin, (cuuint64_t)a.w, (cuuint64_t)a.h, (cuuint64_t)images};
  const cuuint64_t strides[3] = {(cuuint64_t)(a.pitch_w ? a.pitch_w : a.cin),
                                 (cuuint64_t)(a.pitch_h ? a.pitch_h : (long long)a.cin * a.w), (cuuint64_t)image};
  const int lower[2] = {-a.pad, -a.pad};
  const int pad_after = a.pad + a.pad_after_delta;
  const int upper[2] = {pad_after - (a.kw - 1), pad_after - (a.kh - 1)};
  const cuuint32_t estr[4] = {1, (cuuint32_t)a.stride, (cuuint32_t)a.stride, 1};
  return g_encode_im2col(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(a.in), dims, strides, lower, upper,
                         (cuuint32_t)bkb, (cuuint32_t)pixels, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(bkb),
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace
