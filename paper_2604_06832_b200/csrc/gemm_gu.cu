// Gate and up projection of a decode forward with the SwiGLU between them: act = silu(x wg^T) * (x wu^T), up to 64 rows.
//
// The weights are most of a layer's bytes, so this launch is laid out for streaming: one CTA per SM, each with an equal share of
// the features (F of the gate matrix and the same F of the up matrix) over the whole depth.  The share is the MMA's N, which goes in
// steps of 8 features where the MMA's M goes in steps of 128: 11008 features are 138 equal CTAs instead of 172 tiles
// on 148 SMs.  The rows (all planes of them: bf16 hi + lo, or three e5m2 planes) are the MMA's M; they come from L2 once
// per SM, all planes in one box.  All shared memory is one ring: 7 stages of 28 KB at 32 rows of bf16 (with 4 the launch takes 3 us longer).
// What bounds it is memory: of the 90 MB of the 3B shape's gate and up at 32 rows 34 MB lie in L2 (brought by the attention) and 20 MB in the
// rings when its predecessor ends; 14 us from there, 0.9 of them the hand-over, 2 the epilogue.  A layer's gate / up and down launches together,
// with 64-feature tiles : now: 26.9 : 23.0 us at 32 rows, 34.3 : 26.2 at 64 (7B fp8, 64 rows 48.8 : 45.9).
// Every mbarrier wait is bounded (see gemm_tc.cu).
#include "kernels.h"
#include "tc_ptx.cuh"

namespace fdk {

// warp 0 TMA producer of the weights, 1 MMA issuer, 2 TMA producer of the rows, 3.. epilogue
constexpr int GU_EPI_WARPS = 12, GU_EPI = 32 * GU_EPI_WARPS, GU_THREADS = 96 + GU_EPI;
constexpr int GU_STAGES = 10;
enum { GU_BF16 = 0, GU_FP8 = 1, GU_A8 = 2 };      // operand kinds, as TC_KIND_* of gemm_tc.cu

struct GuParams {
  CUtensorMap tm_w[2], tm_x;
  NextWeights next;
  const float* scale[2];
  int m, mp, planes, inter, f, kblocks, kb_elems, stages, w_bytes, x_bytes, tmem_cols;
  void* act; size_t act_lo_off; int act_fmt;
  const float* ssq_in; int nt; float inv_h, eps;
  const float* x_scale; float* amax_out;
  int* status;
  KStamp* stamp;
};

template <int KIND>
__global__ void __launch_bounds__(GU_THREADS, 2) gemm_gu_kernel(const __grid_constant__ GuParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[3 * GU_STAGES + 2];
  __shared__ uint32_t tmem_slot_s;
  __shared__ int abort_s, amax_s[64];
  __shared__ float rs[64], sc[2][128];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bar0 = smem_u32(bars);
  auto wfull = [&](int s) { return bar0 + 8u * s; };
  auto xfull = [&](int s) { return bar0 + 8u * (GU_STAGES + s); };
  auto empty = [&](int s) { return bar0 + 8u * (2 * GU_STAGES + s); };
  const uint32_t tfull = bar0 + 8u * (3 * GU_STAGES), mma_done = tfull + 8u;
  volatile int* abort_flag = &abort_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stage_bytes = p.x_bytes + p.w_bytes;      // the rows first: the MMA reads 128 of them, whatever follows the real ones

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) { mbar_init(wfull(s), 1); mbar_init(xfull(s), 1); mbar_init(empty(s), 1); }
    mbar_init(tfull, 1); mbar_init(mma_done, 1);
    stamp_start(p.stamp);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot_s)), "r"(p.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *(volatile uint32_t*)&tmem_slot_s;
  pdl_trigger();                        // (holding its tensor memory: see gemm_tc.cu)
  const int tile = blockIdx.x, lanes = p.planes * p.mp, n = 2 * p.f;      // rows of the MMA in use, features

  if (warp == 0 || warp == 2) {
    // One thread for the weights, one for the rows: every wait and every load costs its thread some 100 clocks.  The weights do not
    // depend on the predecessor kernel: their first ring is in flight before it has ended.
    if (elect_one()) {
      const bool weights = warp == 0;
      const uint64_t pol = weights ? policy_evict_first() : policy_evict_last();
      bool ok = may_issue(p.status, abort_flag);
      if (!weights) {
        pdl_wait();
        stamp_released(p.stamp);
      }
      int s = 0, issued = 0;
      uint32_t phase = 1;
      // every CTA starts at another k-block: their rows are the same few L2 lines
      int kb = (int)((blockIdx.x * 7u) % (unsigned)p.kblocks);
      for (int j = 0; j < p.kblocks; ++j) {
        if (!ok || !mbar_wait(empty(s), phase, abort_flag)) { ok = false; break; }
        const uint32_t dst = base + s * stage_bytes;
        if (weights) {
          mbar_expect_tx(wfull(s), p.w_bytes);
          tma_load_2d(dst + p.x_bytes, &p.tm_w[0], wfull(s), kb * p.kb_elems, tile * p.f, pol);
          tma_load_2d(dst + p.x_bytes + p.w_bytes / 2, &p.tm_w[1], wfull(s), kb * p.kb_elems, tile * p.f, pol);
        } else {
          mbar_expect_tx(xfull(s), p.x_bytes);
          if (KIND == GU_A8) tma_load_2d(dst, &p.tm_x, xfull(s), kb * p.kb_elems, 0, pol);
          else tma_load_3d(dst, &p.tm_x, xfull(s), kb * p.kb_elems, 0, 0, pol);
        }
        ++issued;
        if (++kb == p.kblocks) kb = 0;
        if (++s == p.stages) { s = 0; phase ^= 1u; }
      }
      if (weights) {
        // Memory would idle from here through the epilogue, the hand-over and the next launch's start: it brings part of the
        // next launch's weights into L2 instead.
        if (ok) ask_for_next(p.next, blockIdx.x, gridDim.x);
        pdl_wait();
      }
      if (!ok) atomicCAS(p.status, 0, ST_PRODUCER);
      if (*abort_flag)      // (see linger) the last copies into each stage
        for (int i = max(0, issued - p.stages); i < issued; ++i)
          mbar_drain(weights ? wfull(i % p.stages) : xfull(i % p.stages), (uint32_t)(i / p.stages) & 1u);
    }
    __syncwarp();
  } else if (warp == 1) {
    // A = rows (e5m2 planes: format code 1 of the A side), B = weights.  One thread runs the whole loop: behind an election per
    // k-block four MMAs took 510 clocks with their waits, from one thread 340.
    const uint32_t idesc = KIND == GU_BF16 ? umma_idesc_bf16(n) : (umma_idesc_e4m3(n) | (KIND == GU_FP8 ? 1u << 7 : 0u));
    if (elect_one()) {
      bool ok = true;
      int s = 0;
      uint32_t phase = 0, off = 0;
      const uint64_t ad0 = umma_desc_sw128(base), bd0 = umma_desc_sw128(base + p.x_bytes);
#pragma unroll 1
      for (int j = 0; j < p.kblocks; ++j) {
        if (!(mbar_wait(wfull(s), phase, abort_flag) && mbar_wait(xfull(s), phase, abort_flag))) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t adesc = ad0 + off, bdesc = bd0 + off;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {      // 32 bytes of k per instruction
          const uint32_t acc = (j > 0 || kk > 0) ? 1u : 0u;
          if (KIND == GU_BF16) umma_bf16(tmem, adesc + 2u * kk, bdesc + 2u * kk, idesc, acc);
          else umma_f8(tmem, adesc + 2u * kk, bdesc + 2u * kk, idesc, acc);
          // rows 128 .. of the planes (fp8 weights, more than 40 rows)
          if (KIND == GU_FP8 && lanes > 128) umma_f8(tmem + 256, adesc + 1024u + 2u * kk, bdesc + 2u * kk, idesc, acc);
        }
        umma_commit(empty(s));
        off += (uint32_t)stage_bytes >> 4;
        if (++s == p.stages) { s = 0; phase ^= 1u; off = 0; }
      }
      if (ok) umma_commit(tfull);
      else atomicCAS(p.status, 0, ST_MMA);
      if (*abort_flag) {
        umma_commit(mma_done);
        mbar_drain(mma_done, 0);
        linger();
      }
    }
    __syncwarp();
  } else {
    const int q = warp & 3, w = warp - 3, t = (int)threadIdx.x - 96;
    pdl_wait();      // the row statistics, and act, which the kernel before last may have been reading
    // folded RMSNorm: two threads add up a row's partial sums
    if (t < 128) {
      float s = 0.f;
      const int r = t >> 1;
      if (r < p.m)
        for (int i = t & 1; i < p.nt; i += 2) s += __ldcg(p.ssq_in + (size_t)r * p.nt + i);
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      if ((t & 1) == 0) rs[r] = rsqrtf(s * p.inv_h + p.eps) * (KIND == GU_A8 && r < p.m ? __ldcg(p.x_scale + r) : 1.f);
      if (t < 64) amax_s[t] = 0;
    }
    if (p.scale[0])
      for (int i = t; i < n; i += GU_EPI) {
        const int side = i >= p.f, j = side ? i - p.f : i, c = tile * p.f + j;
        sc[side][j] = c < p.inter ? p.scale[side][c] : 0.f;
      }
    bool ok = mbar_wait(tfull, 0, abort_flag);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // the accumulators, turned to [feature][row of the MMA] (all MMAs are complete: the ring is free)
    const int stride = lanes | 1;
    float* turned = reinterpret_cast<float*>(smem_raw + (base - smem_u32(smem_raw)));
    for (int pass = 0; pass * 128 < lanes; ++pass) {
      const int row = pass * 128 + q * 32 + lane;
      if (pass * 128 + q * 32 >= lanes) continue;           // uniform over the warp
      const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + pass * 256;
      for (int c = (w >> 2) * 16; c < n; c += GU_EPI_WARPS * 4) {      // GU_EPI_WARPS / 4 warps share a lane quarter
        float v[16];
        tmem_ld16(taddr + c, v);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (row < lanes && ok) {
#pragma unroll
          for (int i = 0; i < 16; ++i) turned[(c + i) * stride + row] = v[i];
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    ok = named_barrier_and<GU_EPI>(ok);
    // 8 rows x 4 groups of 8 features per warp and step: no bank conflicts (the stride is odd), 64 bytes of a row side by side
    const int groups = p.f / 8, gblocks = (groups + 3) / 4, blocks = (p.mp / 8) * gblocks;
    for (int b = w; ok && b < blocks; b += GU_EPI_WARPS) {
      const int row = (b / gblocks) * 8 + (lane & 7), grp = (b % gblocks) * 4 + (lane >> 3);
      const int col = tile * p.f + grp * 8;
      if (grp >= groups || row >= p.m || col >= p.inter) continue;
      const float r = rs[row];
      float val[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float* a = turned + (grp * 8 + i) * stride + row;
        const float* b_ = a + p.f * stride;
        float g = a[0], u = b_[0];
        if (KIND == GU_BF16) { g += a[p.mp]; u += b_[p.mp]; }      // low-order plane
        if (KIND == GU_FP8) {                                      // x = p0 + p1 / 4 + p2 / 128
          g += fmaf(a[2 * p.mp], 0.0078125f, a[p.mp] * 0.25f);
          u += fmaf(b_[2 * p.mp], 0.0078125f, b_[p.mp] * 0.25f);
        }
        if (p.scale[0]) { g *= sc[0][grp * 8 + i]; u *= sc[1][grp * 8 + i]; }
        val[i] = silu_mul(g * r, u * r);
      }
      const size_t idx = (size_t)row * p.inter + col;
      store_act4(p.act, p.act_lo_off, idx, make_float4(val[0], val[1], val[2], val[3]), p.act_fmt);
      store_act4(p.act, p.act_lo_off, idx + 4, make_float4(val[4], val[5], val[6], val[7]), p.act_fmt);
      if (KIND == GU_A8) {
        // maximum of |act| as stored (f16): non-negative values, whose bit patterns order like integers
        float mx = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) mx = fmaxf(mx, fabsf(__half2float(__ushort_as_half(f16_bits_sat(val[i])))));
        atomicMax(&amax_s[row], __float_as_int(mx));
      }
    }
    if (KIND == GU_A8) {
      asm volatile("bar.sync 1, %0;" ::"n"(GU_EPI) : "memory");
      if (ok && t < p.m && amax_s[t] > 0) atomicMax(reinterpret_cast<int*>(p.amax_out) + t, amax_s[t]);
    }
    if (!ok) {
      if (lane == 0) atomicCAS(p.status, 0, ST_EPILOGUE);
      linger();
    }
  }

  // ---- teardown: every thread arrives here, whatever happened ----
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem_cols) : "memory");
  }
  if (threadIdx.x == 0) stamp_end(p.stamp);
}

template <int KIND>
static cudaError_t gu_launch_t(const GuParams& p, int grid, size_t smem, cudaStream_t st) {
  static bool attr_set[MAX_DEVICES] = {};
  cudaError_t e = ensure_dynamic_smem(gemm_gu_kernel<KIND>, 224 * 1024, attr_set);
  if (e != cudaSuccess) return e;
  return launch_pdl(gemm_gu_kernel<KIND>, dim3(grid), dim3(GU_THREADS), smem, st, p);
}

// The launch for g: shares and shared memory.  False: g is left to gemm_tc_kernel.
struct GuPlan { int kind, f, mp, planes, kblocks, stages; size_t smem; };
static bool gu_plan(const TcGroup& g, GuPlan* pl) {
  pl->kind = g.a8 ? GU_A8 : (g.fp8 ? GU_FP8 : GU_BF16);
  // fp8 weights, 41 to 48 rows: more than 128 lanes take a second MMA, which eats up what the shares gain, while the 64-feature tiles still
  // have three stages (two from 49 rows on).  us a step, shares : tiles, 8 layers of the 7B shape: 32 rows 658 : 658, 33 rows 682 : 694, 40 rows
  // 697 : 719, 41 rows 740 : 722, 44 rows 750 : 727, 48 rows 767 : 742, 49 rows 815 : 830, 56 rows 805 : 830, 64 rows 855 : 866.
  // Everywhere else the shares are as fast or faster: 12 layers of the 3B shape, 4, 16, 32, 64 rows: 679, 696, 731, 835 : 683, 707, 763, 923.
  if (pl->kind == GU_FP8 && g.m > 40 && g.m <= 48) return false;
  // A few MB of weights and few rows: everything is latency, and the smaller CTAs of the tiles start sooner.  us a step, shares : tiles: 12 layers of
  // hidden 512, intermediate 1376 in bf16 (2.8 MB): 2 rows 360 : 349, 4 rows 367 : 352, 8 rows 378 : 365, 16 rows 366 : 366, 32 rows 422 : 454;
  // of 1024 and 2816 in fp8 (5.8 MB): 391 : 374, 391 : 379, 396 : 374, 405 : 387, 427 : 462; of 1536 and 8960 in bf16 (55 MB): 2 rows 480 : 485,
  // 8 rows 503 : 510.
  if (g.m <= 8 && (size_t)g.n[0] * g.k * (g.fp8 ? 2 : 4) <= (8u << 20)) return false;
  pl->f = ((ceil_div(g.n[0], sm_count()) + 7) / 8) * 8;
  if (pl->f > 128) return false;        // N = 256 at most
  pl->mp = ((g.m + 7) / 8) * 8; pl->planes = pl->kind == GU_FP8 ? 3 : (pl->kind == GU_A8 ? 1 : 2);
  pl->kblocks = ceil_div(g.k, g.fp8 ? 2 * TC_BK : TC_BK);
  const int lanes = pl->planes * pl->mp, n = 2 * pl->f, stage = (n + lanes) * 128;
  pl->stages = 221 * 1024 / stage;
  if (pl->stages > GU_STAGES) pl->stages = GU_STAGES;
  if (pl->stages > pl->kblocks) pl->stages = pl->kblocks;
  // the ring; the rows that the MMA reads behind the last stage's real ones; the turned accumulators
  size_t smem = (size_t)pl->stages * stage;
  const size_t reach = (size_t)(pl->stages - 1) * stage + (lanes > 128 ? 32768 : 16384), turned = (size_t)n * (lanes | 1) * 4;
  if (smem < reach) smem = reach;
  if (smem < turned) smem = turned;
  pl->smem = smem + 1024;
  return pl->smem <= 224 * 1024;
}

bool gemm_gu_supported(const TcGroup& g) {
  GuPlan pl;
  return g.m >= 1 && g.m <= 64 && gu_plan(g, &pl);
}

cudaError_t gemm_gu_launch(const TcGroup& g, const TcOut& o, const void* next, int next_n, int next_k, cudaStream_t st) {
  GuParams p;
  GuPlan pl;
  memset(&p, 0, sizeof(p));
  const int inter = g.n[0];
  if (g.m < 1 || g.m > 64 || g.n_mats != 2 || g.n[1] != inter || inter % 8 || !o.ssq_in || !gu_plan(g, &pl)) return cudaErrorInvalidValue;
  if (pl.kind == GU_A8 ? (!o.x_scale || !o.amax_out) : !g.x_lo) return cudaErrorInvalidValue;
  p.f = pl.f; p.m = g.m; p.mp = pl.mp; p.planes = pl.planes; p.inter = inter; p.stages = pl.stages; p.kblocks = pl.kblocks;
  p.kb_elems = g.fp8 ? 2 * TC_BK : TC_BK;
  p.w_bytes = 2 * p.f * 128; p.x_bytes = p.planes * p.mp * 128;
  p.scale[0] = g.scale[0]; p.scale[1] = g.scale[1];
  p.act = o.act; p.act_lo_off = o.act_lo_off; p.act_fmt = o.act_fmt;
  p.ssq_in = o.ssq_in; p.nt = o.nt_in; p.inv_h = o.hidden > 0 ? 1.f / (float)o.hidden : 0.f; p.eps = o.eps;
  p.x_scale = o.x_scale; p.amax_out = o.amax_out; p.status = o.status; p.stamp = o.stamp;
  const int lanes = p.planes * p.mp, n = 2 * p.f;
  p.tmem_cols = lanes > 128 ? 512 : (n <= 32 ? 32 : (n <= 64 ? 64 : (n <= 128 ? 128 : 256)));
  const int xkind = g.fp8 ? TM_E4M3_128 : TM_BF16;
  if (pl.kind == GU_A8 ? !make_tmap(&p.tm_x, g.x, g.m, g.k, p.mp, xkind)
                       : !make_tmap_planes(&p.tm_x, g.x, g.m, g.k, p.planes, (const char*)g.x_lo - (const char*)g.x, p.mp, xkind))
    return cudaErrorInvalidValue;
  for (int i = 0; i < 2; ++i)
    if (!make_tmap(&p.tm_w[i], g.w[i], inter, g.k, p.f, xkind)) return cudaErrorInvalidValue;
  // Part of the next launch's weights (NextWeights, every third pair), up to 32 rows.  us a step without : with, a process each: 3B shape, 12
  // layers: 4 rows 672 : 672, 16 rows 706 : 701, 24 rows 723 : 717, 32 rows 739 : 734, 33 rows 754 : 754, 48 rows 782 : 780, 64 rows 842 : 839
  // (7B shape in bf16, 6 layers, 48 rows 865 : 873).  7B shape, 8 layers, fp8: 4 rows 597 : 588, 16 rows 610 : 600, 32 rows 648 : 644, 33 rows
  // 684 : 686, 40 rows 705 : 707; W8A8: 8 rows 633 : 625, 16 rows 646 : 645, 32 rows 697 : 696, 33 rows 706 : 709, 48 rows 722 : 730.
  if (next && g.m <= 32 && !next_weights(&p.next, next, nullptr, next_n, next_k, g.fp8, 3)) return cudaErrorInvalidValue;
  const int grid = ceil_div(inter, p.f);
  return pl.kind == GU_A8 ? gu_launch_t<GU_A8>(p, grid, pl.smem, st)
                          : (pl.kind == GU_FP8 ? gu_launch_t<GU_FP8>(p, grid, pl.smem, st) : gu_launch_t<GU_BF16>(p, grid, pl.smem, st));
}

}  // namespace fdk
