// PTX wrappers shared by the tcgen05 / TMA kernels (sm_100a): mbarriers with bounded waits, 2-D bulk
// tensor loads, shared-memory matrix descriptors, tcgen05.mma / commit / ld.
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace fdk {

constexpr int TC_BM = 128;       // weight rows per tile (MMA M)
constexpr int TC_BK = 64;        // bf16 elements per k-block: 128 bytes = one swizzle atom row
constexpr long long TC_TIMEOUT = 1ll << 28;  // clock cycles (~0.14 s) before a wait gives up

// ---- PTX wrappers -------------------------------------------------------------------------------
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
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// The same test, but the thread may be suspended by the hardware for up to `ns` nanoseconds while the phase is not
// complete: a waiting thread then takes no issue slots from the warps that share its scheduler.
__device__ __forceinline__ bool mbar_try_wait_suspend(uint32_t bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(ns)
      : "memory");
  return ok != 0;
}
// Bounded wait of one thread.  Returns false when the wait gave up (timeout here, or another thread's abort).
// The lanes of a warp may see different ends of one wait: another role's abort or the clock limit can fall just as the barrier
// completes.  So a warp that goes on to warp-wide instructions (elect.sync, tcgen05.ld / st, shuffles, votes) never leaves its loop
// for a wait that gave up: the lane notes it (ok = ok && mbar_wait(...): it waits for nothing any more), all lanes run the loop to
// its end, and what is issued or announced to other roles depends on ok.  (A vote behind every wait was as safe and cost 0.4 % of
// a decode forward and 3 % of an fp8 prompt.)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
    if (mbar_try_wait_suspend(bar, parity, 20000u)) return true;
    if (*abort_flag) return false;
    if (clock64() - t0 > TC_TIMEOUT) { *abort_flag = 1; return false; }
  }
}
// What a CTA must not leave behind (bulk copies, MMAs): a bounded wait that no abort ends.
__device__ __forceinline__ void mbar_drain(uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity) && clock64() - t0 < TC_TIMEOUT) {}
}
// No CTA leaves with a copy or an MMA in flight, whoever gives up.  A producer or MMA thread that finds the abort flag raised when its loop has
// ended (no wait of its own may have failed: where all k-blocks fit into the ring a producer waits for nothing) drains what it issued.  Where
// the flag is raised later, all of that has been issued before: whoever gives up lingers for a time (0.5 ms) that copies and MMAs need many
// times over, before it comes to the CTA's last barrier.  (Waiting in every CTA, or reading the flag behind the last barrier, where the code is
// fetched in vain, cost 0.2 to 1 % of a decode step.)
__device__ __forceinline__ void linger() {
  const long long t0 = clock64();
  while (clock64() - t0 < (1ll << 20)) {}
}
// The host-set test hook (status[1]; written by the host only, never by a kernel of the chain, so it may be read before the wait for
// the predecessor).  1: the abort flag is raised, which every other role's first wait sees, and the producer is to issue nothing
// (returns false): all leave by the path a timed-out wait takes.  2: the flag is raised, the others are given the time to see it, and
// the producer goes on as one that has waited for nothing yet.  Only the producers pay for the read.
__device__ __forceinline__ bool may_issue(const int* status, volatile int* abort_flag) {
  const int hook = status ? *reinterpret_cast<const volatile int*>(status + 1) : 0;
  if (hook == 0) return true;
  *abort_flag = 1;
  const long long t0 = clock64();
  while (hook == 2 && clock64() - t0 < (1ll << 17)) {}
  return hook == 2;
}
// Barrier 1 of N threads that also tells every thread whether all of them came with `ok`.
template <int N>
__device__ __forceinline__ bool named_barrier_and(bool ok) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(r) : "r"((uint32_t)ok), "n"(N) : "memory");
  return r != 0;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
      ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, int c2, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;"
      ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "l"(pol)
      : "memory");
}
// asks for a box of a 2-D tensor in L2
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* tm, int c0, int c1) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(tm), "r"(c0), "r"(c1) : "memory");
}
// Part of the weights that a later launch streams, asked for in L2 while memory would idle: of every 64 rows of one or two
// matrices of `kblocks` k-blocks every step-th pair of k-blocks from the first on (step 3, 32 k-blocks: 6 of 16 pairs, 37.5 %; one or
// two k-blocks: all).  units (pairs of all rows) = 0: nothing.
struct NextWeights {
  CUtensorMap tm[2];
  int mats, units, row_blocks, step, kblocks, kb_elems;
};
// one thread's share: units first, first + stride, ...
__device__ __forceinline__ void ask_for_next(const NextWeights& n, int first, int stride) {
  for (int u = first; u < n.units; u += stride) {
    const int pair = u / n.row_blocks, row = (u - pair * n.row_blocks) * 64, kb = pair * 2 * n.step;
    for (int i = 0; i < n.mats; ++i) {
      tma_prefetch_2d(&n.tm[i], kb * n.kb_elems, row);
      if (kb + 1 < n.kblocks) tma_prefetch_2d(&n.tm[i], (kb + 1) * n.kb_elems, row);
    }
  }
}
bool next_weights(NextWeights* n, const void* w0, const void* w1, int rows, int k, bool fp8, int step);
__device__ __forceinline__ void tma_load_2d_plain(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
               ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1)
               : "memory");
}
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
// True in one lane of a converged warp, the same one every time.  MMAs and commits are issued inside `if (elect_one())`: one thread is
// then known to execute them.  Inside `if (lane == 0)` each costs some 100 clocks of the issuing thread; an election in front of a group
// of MMAs costs some 250.  So where that is not hidden, the whole loop, waits included, runs in one elected thread (gemm_gu.cu,
// attention.cu, prefill_attn.cu); gemm_tc.cu (two CTAs per SM) and prefill_gemm.cu (N = 256) elect per k-block, which costs them nothing.
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r != 0;
}
// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows 128 bytes apart, groups
// of 8 rows 1024 bytes apart (stride-dimension byte offset), descriptor version 1 (sm_100).
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;                 // leading-dimension offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;       // stride-dimension offset
  d |= (uint64_t)1 << 46;                 // version
  d |= (uint64_t)2 << 61;                 // SWIZZLE_128B
  return d;
}
// The same for an MN-major operand: rows are 8-element groups of k, 128 bytes = 64 elements of the M / N dimension, whose
// blocks of 64 lie `block_bytes` apart.
__device__ __forceinline__ uint64_t umma_desc_sw128_mn(uint32_t saddr, uint32_t block_bytes) {
  return (umma_desc_sw128(saddr) & ~((uint64_t)0x3FFF << 16)) | ((uint64_t)(block_bytes >> 4) << 16);
}
// Instruction descriptor, kind::f16: D = f32, A = B = bf16, both K-major, M = m, N = n.
__device__ __forceinline__ uint32_t umma_idesc_bf16(int n, int m = TC_BM) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
// The same with A = B = f16.
__device__ __forceinline__ uint32_t umma_idesc_f16(int n, int m = TC_BM) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
// kind::f16 covers f16 x f16 and bf16 x bf16 alike; the instruction descriptor names the operand type.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
// A operand from tensor memory (lane = row, two 16-bit elements of k per column)
__device__ __forceinline__ void umma_f16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
// kind::f8f6f4 with both operands e4m3 (format code 0), fp32 accumulation, K-major; one instruction covers 32 k
__device__ __forceinline__ uint32_t umma_idesc_e4m3(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TC_BM >> 4) << 24);
}
// the same with B = e5m2 (format code 1): weights are the A operand, the planes of the rows the B operand
__device__ __forceinline__ uint32_t umma_idesc_e4m3_e5m2(int n) { return umma_idesc_e4m3(n) | (1u << 10); }
__device__ __forceinline__ void umma_f8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};"
      ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// ---- CTA pairs (tcgen05 cta_group::2): two CTAs of a cluster, rank 0 issues the MMAs of both ---------------------
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}
// address of the same shared-memory location in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Arrival on the peer's barrier.  Default (CTA) scope on purpose: it hands over shared-memory tiles that fence.proxy.async
// has already made visible to the tensor core, or nothing but the arrival itself; with .release.cluster every arrival waited
// for a memory barrier (widening an fp8 tile took 1800 clocks instead of the 512 of its MMAs).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t mapped) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(mapped) : "memory");
}
// 2-D TMA load into this CTA's shared memory whose bytes are counted on the pair leader's barrier at the same offset
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
               ::"r"(dst), "l"(tm), "r"(bar & 0xFEFFFFFFu), "r"(c0), "r"(c1)
               : "memory");
}
__device__ __forceinline__ void umma_f16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
// arrives on the barrier at this offset in both CTAs once the MMAs issued so far have completed
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"((unsigned short)3) : "memory");
}

// sixteen e4m3 bytes -> sixteen f16 (exact: every e4m3 value, subnormals included, is an f16 value)
__device__ __forceinline__ void e4m3x16_to_f16(const uint4& in, uint4& lo, uint4& hi) {
  const uint32_t w[4] = {in.x, in.y, in.z, in.w};
  uint32_t o[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int hsel = 0; hsel < 2; ++hsel) {
      const unsigned short two = (unsigned short)(hsel ? (w[i] >> 16) : (w[i] & 0xffffu));
      asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(o[2 * i + hsel]) : "h"(two));
    }
  }
  lo = make_uint4(o[0], o[1], o[2], o[3]);
  hi = make_uint4(o[4], o[5], o[6], o[7]);
}

// A warp's 32 x W block of values, thread = row, turned round through shared memory (32 * W floats of the warp's own,
// 16-byte pieces XOR-swizzled, no bank conflicts either way): lane l gets columns 4 (l % (W/4)) .. + 3 of the rows
// l / (W/4) + i * 128 / W, so that the warp's accesses to global memory are whole sectors of few rows instead of 16 bytes
// of 32 rows (which made the epilogue as long as the main loop of a 2048-deep tile).
template <int W>
__device__ __forceinline__ void turn(uint32_t buf, int lane, const float* v, float4* w) {
  constexpr int PR = W / 4, RI = 32 / PR;       // 16-byte pieces per row, rows per step
  auto at = [&](int r, int c) { return buf + (uint32_t)((r * PR + (c ^ (W == 32 ? (r & 7) : ((r >> 1) & 3)))) << 4); };
  __syncwarp();
#pragma unroll
  for (int c = 0; c < PR; ++c)
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at(lane, c)), "f"(v[4 * c]), "f"(v[4 * c + 1]), "f"(v[4 * c + 2]), "f"(v[4 * c + 3]) : "memory");
  __syncwarp();
#pragma unroll
  for (int i = 0; i < W / 4; ++i)
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(w[i].x), "=f"(w[i].y), "=f"(w[i].z), "=f"(w[i].w) : "r"(at(lane / PR + i * RI, lane % PR)) : "memory");
}
}  // namespace fdk
