// Small-M weight-streaming GEMM for sm_100a: y[m, n] = sum_k x[m, k] w[n, k], m <= 64.
//
// The weight matrix is the MMA "A" operand (128 output features per tile fill the tensor-core M
// dimension), the m activation rows are the MMA "N" dimension (padded to 16/32/48/64), so a CTA
// streams 128 x K weights once while the tiny activation tile comes from L2.  Weights and
// activations are staged by TMA (128-byte swizzle, K-major) into a ring of shared-memory stages;
// one elected thread issues tcgen05.mma with fp32 accumulators in tensor memory (two accumulator
// buffers, so the epilogue of one work item overlaps the mainloop of the next); four epilogue warps
// read the accumulators with tcgen05.ld.  CTAs are persistent over a static round-robin list of
// work items (tile, K-split).  bf16 weights: the activations arrive as two bf16 planes, hi = bf16(v) and
// lo = bf16(v - hi); both land side by side in the stage and form ONE MMA operand of twice the rows, so every streamed
// weight tile is read from shared memory once and multiplied by both; the epilogue adds the two halves of the
// accumulator.  The activation side of the product thus carries ~16 significant bits at no extra HBM traffic.
// FP8-E4M3 weights: the byte tile is the MMA operand as it lands.  The rows are f16 values, stored as three planes of
// e5m2 bytes whose weighted sum they are (XF_E5M2X3), again one MMA operand (of three times the rows, kind::f8f6f4, fp32
// accumulation); the epilogue adds the three parts of the accumulator and applies the per-channel scales.  (Widening the
// bytes to f16 in converter warps made the converters the bottleneck: 7B gate/up 34.5 us a layer.)
// Every mbarrier wait is bounded: on a timeout the CTA records an
// error code in a status word, drains its own bulk copies, frees its tensor memory and returns.
#include <cuda.h>

#include <map>
#include <mutex>
#include <tuple>

#include "kernels.h"
#include "tc_ptx.cuh"

namespace fdk {

constexpr int TC_THREADS = 192;       // warp 0 TMA producer, warp 1 MMA issuer, warps 2..5 epilogue
constexpr int TC_A_BYTES = TC_BM * TC_BK * 2;   // a bf16 weight tile

enum { TC_ERR_PRODUCER = ST_PRODUCER, TC_ERR_MMA = ST_MMA, TC_ERR_EPILOGUE = ST_EPILOGUE };

struct TcParams {
  CUtensorMap tm_w[3];  // weight matrices, box {64 k, 64 rows}
  CUtensorMap tm_x;     // activations (hi plane, or the only one), box {64 k, m_pad rows}
  CUtensorMap tm_xl;    // lo plane of the activations (has_lo); fp8: second plane
  CUtensorMap tm_x3;    // fp8: third plane
  int has_lo;
  int n_out[3];         // rows (output features) of each matrix
  int tile_begin[4];    // first tile of each matrix; [n_mats] = total tiles
  int out_col[3];       // column of each matrix's first feature in the output row
  const float* scale[3];
  int n_mats, kblocks, splits, kb_per_split, m, mode;
  float* part;          // [splits][m][ldp]     (PARTIAL)
  int ldp;
  float* y;             // [m][ldy]             (LOGITS)
  int ldy;
  void* act;            // [m][inter]           (SWIGLU), stored as act_fmt (XF_*), lo plane act_lo_off elements on
  size_t act_lo_off;
  int act_fmt, inter;
  // RMSNorm folded into the consumer: x holds bf16(h * gain); the per-row factor rsqrt(mean(h^2) + eps)
  // is applied to the accumulators.  ssq_in[row][nt_in] holds partial sums of h^2 (null: factor 1).
  const float* ssq_in;
  int nt_in;
  float inv_h, eps;
  // LOGITS mode: per (tile, lane quarter, row) softmax statistics of the 32 columns a warp holds, the
  // mask token's column excluded: (max, sum exp(l - max), argmax column)
  float4* stats;        // [tiles * 4][m]
  int mask_id, write_logits;
  int* status;          // device words: [0] set non-zero when a wait timed out; [1] read at start: non-zero makes
                        // every role take its give-up path at once (a host-set test hook for that path)
  KStamp* stamp;        // in-chain timing of this launch (null: off)
  // TC_KIND_A8: x_scale[row] = the factor of the row's e4m3 codes.  SWIGLU mode also raises amax_out[row] (atomic maximum;
  // zero before the launch) to the maximum of |act[row]| as stored, for whoever quantises `act`.
  const float* x_scale;
  float* amax_out;
};

// Operand kinds of the kernel:
//   TC_KIND_BF16: bf16 weights x bf16 hi/lo activation planes
//   TC_KIND_FP8 : e4m3 weights x three e5m2 planes of the activations; a k-block is 128 elements
//   TC_KIND_A8  : e4m3 weights x rows of e4m3 codes with one factor per row (W8A8, Sec. 3.4 "System integration"); a k-block
//                 is 128 elements, both byte tiles are MMA operands as they land.  (Quantising the rows in warps of this kernel,
//                 which had to wait for the row maxima first and then stood between every stage and its MMA, cost 4 us in each of
//                 a layer's four projections.)
enum { TC_KIND_BF16 = 0, TC_KIND_FP8 = 1, TC_KIND_A8 = 2 };

template <int M_PAD, int KIND>
struct TcSmem {
  static constexpr bool FP8 = KIND == TC_KIND_FP8, A8 = KIND == TC_KIND_A8;
  static constexpr int STAGES = A8 ? (M_PAD <= 32 ? 5 : 4) : (FP8 ? (M_PAD <= 16 ? 4 : (M_PAD <= 48 ? 3 : 2)) : (M_PAD <= 32 ? 4 : 3));   // two CTAs per SM must fit
  static constexpr int KB_ELEMS = (A8 || FP8) ? 2 * TC_BK : TC_BK;     // k per stage
  static constexpr int W_BYTES = TC_A_BYTES;                           // weight tile
  static constexpr int B_BYTES = M_PAD * 128;                          // one activation plane
  static constexpr int X_PLANES = FP8 ? 3 : (A8 ? 1 : 2);              // e5m2 planes; bf16 hi + lo; codes
  static constexpr int STAGE_BYTES = W_BYTES + X_PLANES * B_BYTES;
  static constexpr int EX_OFF = STAGES * STAGE_BYTES;                  // SwiGLU epilogue: gate/up exchange
  static constexpr int EX_ROWS = KIND != TC_KIND_BF16 ? 16 : 32;       // rows that pass through it per round
  static constexpr int EX_ROUNDS = (M_PAD + EX_ROWS - 1) / EX_ROWS;
  static constexpr int EX_BYTES = (M_PAD / EX_ROUNDS) * 256;
  static constexpr int BAR_OFF = EX_OFF + EX_BYTES;
  static constexpr int RS_OFF = BAR_OFF + 256;                         // the rows' folded norm factors
  static constexpr int TOTAL = RS_OFF + 256 + 1024;                    // + alignment slack
};

template <int M_PAD, int KIND>
__global__ void __launch_bounds__(TC_THREADS) gemm_tc_kernel(const __grid_constant__ TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  using L = TcSmem<M_PAD, KIND>;
  constexpr bool A8 = KIND == TC_KIND_A8;
  constexpr bool W8 = KIND != TC_KIND_BF16;        // weight bytes: a k-block is 128 elements
  constexpr bool X3 = KIND == TC_KIND_FP8;
  constexpr int TC_STAGES = L::STAGES;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* sm = smem_raw + (base - raw);
  const uint32_t bar0 = base + L::BAR_OFF;
  // barrier slots (8 bytes each): full[S], empty[S], tmem_full[2], tmem_empty[2]
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (TC_STAGES + s); };
  auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * TC_STAGES + a); };
  auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * TC_STAGES + 2 + a); };
  // SwiGLU epilogue, per warp pair pr: exchange buffer written (exw) / read (exr), two arrivals each
  auto exw_bar = [&](int pr) { return bar0 + 8u * (2 * TC_STAGES + 6 + pr); };
  auto exr_bar = [&](int pr) { return bar0 + 8u * (2 * TC_STAGES + 8 + pr); };
  const uint32_t done_bar = bar0 + 8u * (2 * TC_STAGES + 10);      // every MMA of the CTA is complete (after an abort)
  volatile uint32_t* tmem_slot = (volatile uint32_t*)(sm + L::BAR_OFF + 8 * (2 * TC_STAGES + 4));
  volatile int* abort_flag = (volatile int*)(sm + L::BAR_OFF + 8 * (2 * TC_STAGES + 4) + 8);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // two accumulator buffers; each holds the products of plane i in columns [i M_PAD, (i + 1) M_PAD)
  constexpr int ACC_COLS = L::X_PLANES * M_PAD;
  // (one buffer where two would leave no tensor memory for a second CTA on the SM)
  constexpr int NACC = 2 * ACC_COLS <= 256 ? 2 : 1;
  constexpr int TMEM_COLS = (NACC * ACC_COLS <= 32) ? 32 : ((NACC * ACC_COLS <= 64) ? 64 : ((NACC * ACC_COLS <= 128) ? 128 : 256));

  if (threadIdx.x == 0) {
    for (int s = 0; s < TC_STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), 4); }
    for (int pr = 0; pr < 2; ++pr) { mbar_init(exw_bar(pr), 2); mbar_init(exr_bar(pr), 2); }
    mbar_init(done_bar, 1);
    stamp_start(p.stamp);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;
  // Dependents may start only now that this CTA holds its tensor memory: a successor CTA that allocated first and then
  // waited for this grid could otherwise keep it from ever getting any.
  pdl_trigger();

  const int total_tiles = p.tile_begin[p.n_mats];
  const int n_items = total_tiles * p.splits;

  if (warp == 0) {
    // ------------------------------------------------ TMA producer ------------------------------------------------
    if (lane == 0) {
      const uint64_t pol_w = policy_evict_first(), pol_x = policy_evict_last();
      int stage = 0;
      uint32_t phase = 0;
      uint32_t armed = 0;           // bit s: full[s] armed
      uint32_t armed_parity = 0;    // bit s: parity of the last arming
      bool ok = may_issue(p.status, abort_flag);
      bool waited = false;
      int n_pend = 0, pend_stage[TC_STAGES], pend_kb[TC_STAGES];
      const uint32_t stage_tx = L::W_BYTES + (X3 ? 3 : (p.has_lo ? 2 : 1)) * L::B_BYTES;
      auto load_x = [&](int st_, int kb_) {
        const uint32_t dst = base + st_ * L::STAGE_BYTES + L::W_BYTES;
        tma_load_2d(dst, &p.tm_x, full_bar(st_), kb_ * L::KB_ELEMS, 0, pol_x);
        if (X3 || p.has_lo) tma_load_2d(dst + L::B_BYTES, &p.tm_xl, full_bar(st_), kb_ * L::KB_ELEMS, 0, pol_x);
        if (X3) tma_load_2d(dst + 2 * L::B_BYTES, &p.tm_x3, full_bar(st_), kb_ * L::KB_ELEMS, 0, pol_x);
      };
      for (int it = blockIdx.x; it < n_items && ok; it += gridDim.x) {
        const int tile = it % total_tiles, split = it / total_tiles;
        int mi = 0, r0 = 0;
        if (p.mode != TC_MODE_SWIGLU) {
          while (mi + 1 < p.n_mats && tile >= p.tile_begin[mi + 1]) ++mi;
          r0 = (tile - p.tile_begin[mi]) * TC_BM;
        }
        const int kb0 = split * p.kb_per_split;
        const int kb1 = min(p.kblocks, kb0 + p.kb_per_split);
        // Every CTA walks its k-blocks from a different starting point (and wraps): the activation tile of a k-block
        // is the same few L2 lines for all CTAs, and in lockstep they would all ask for them at the same moment.
        const int nkb = kb1 - kb0;
        const int rot = (int)((blockIdx.x * 7u) % (unsigned)nkb);
        for (int j = 0; j < nkb; ++j) {
          const int kb = kb0 + ((j + rot) >= nkb ? j + rot - nkb : j + rot);
          if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag)) { ok = false; break; }
          const uint32_t a_dst = base + stage * L::STAGE_BYTES;
          mbar_expect_tx(full_bar(stage), stage_tx);
          armed |= 1u << stage;
          armed_parity = (armed_parity & ~(1u << stage)) | (phase << stage);
          if (p.mode == TC_MODE_SWIGLU) {
            // 64 features per tile: their gate rows fill TMEM lanes 0..63, their up rows lanes 64..127
            tma_load_2d(a_dst, &p.tm_w[0], full_bar(stage), kb * L::KB_ELEMS, tile * 64, pol_w);
            tma_load_2d(a_dst + L::W_BYTES / 2, &p.tm_w[1], full_bar(stage), kb * L::KB_ELEMS, tile * 64, pol_w);
          } else {
            tma_load_2d(a_dst, &p.tm_w[mi], full_bar(stage), kb * L::KB_ELEMS, r0, pol_w);
            tma_load_2d(a_dst + L::W_BYTES / 2, &p.tm_w[mi], full_bar(stage), kb * L::KB_ELEMS, r0 + 64, pol_w);
          }
          // The weights do not depend on the predecessor kernel: the first ring of weight loads is issued before waiting
          // for it; the activation tiles of those stages follow once it has completed.
          if (waited) {
            load_x(stage, kb);
          } else {
            pend_stage[n_pend] = stage; pend_kb[n_pend] = kb;
            if (++n_pend == TC_STAGES) {
              pdl_wait();
              stamp_released(p.stamp);
              waited = true;
              for (int j = 0; j < n_pend; ++j) load_x(pend_stage[j], pend_kb[j]);
            }
          }
          if (++stage == TC_STAGES) { stage = 0; phase ^= 1u; }
        }
      }
      if (!waited) {
        pdl_wait();
        stamp_released(p.stamp);
        for (int j = 0; j < n_pend; ++j) load_x(pend_stage[j], pend_kb[j]);
      }
      if (!ok) atomicCAS(p.status, 0, TC_ERR_PRODUCER);
      if (*abort_flag)      // (see linger)
        for (int s = 0; s < TC_STAGES; ++s)
          if (armed & (1u << s)) mbar_drain(full_bar(s), (armed_parity >> s) & 1u);
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer --------------------------------------------------
    {
      const uint32_t idesc = A8 ? umma_idesc_e4m3(M_PAD) : (X3 ? umma_idesc_e4m3_e5m2(3 * M_PAD) : umma_idesc_bf16(p.has_lo ? 2 * M_PAD : M_PAD));
      int stage = 0;
      uint32_t phase = 0;
      int local = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < n_items; it += gridDim.x, ++local) {
        const int split = it / total_tiles;
        const int acc = local % NACC;
        const uint32_t acc_phase = (uint32_t)(local / NACC) & 1u;
        ok = ok && mbar_wait(tempty_bar(acc), acc_phase ^ 1u, abort_flag);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * ACC_COLS);
        const int kb0 = split * p.kb_per_split;
        const int kb1 = min(p.kblocks, kb0 + p.kb_per_split);
        for (int kb = kb0; kb < kb1; ++kb) {
          ok = ok && mbar_wait(full_bar(stage), phase, abort_flag);
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a_addr = base + stage * L::STAGE_BYTES;
          const uint64_t adesc = umma_desc_sw128(a_addr);
          const uint64_t bdesc = umma_desc_sw128(a_addr + L::W_BYTES);
          if (elect_one() && ok) {
          if (W8) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)      // 32 bytes of k per instruction
              umma_f8(d_tmem, adesc + 2u * kk, bdesc + 2u * kk, idesc, (kb > kb0 || kk > 0) ? 1u : 0u);
          } else {
#pragma unroll
            for (int kk = 0; kk < TC_BK / 16; ++kk)
              umma_bf16(d_tmem, adesc + 2u * kk, bdesc + 2u * kk, idesc, (kb > kb0 || kk > 0) ? 1u : 0u);
          }
          umma_commit(empty_bar(stage));
          }
          if (++stage == TC_STAGES) { stage = 0; phase ^= 1u; }
        }
        if (elect_one() && ok) umma_commit(tfull_bar(acc));
      }
      if (!ok) atomicCAS(p.status, 0, TC_ERR_MMA);
      if (__any_sync(0xffffffffu, *abort_flag != 0)) {
        if (elect_one()) {
          umma_commit(done_bar);
          mbar_drain(done_bar, 0);
        }
        linger();
      }
    }
  } else {
    // ------------------------------------------------ epilogue warps ----------------------------------------------
    const int q = warp & 3;  // TMEM lane quarter this warp may read
    int local = 0;
    bool ok = true;
    pdl_wait();   // the epilogue reads the predecessor's row statistics and overwrites buffers it may still be reading
    // folded RMSNorm: lane l keeps the factor of rows l and l + 32; broadcast by shuffle where needed.  Two threads add up a
    // row's partial sums, so that the CTA asks for each of them once (they are the same few lines of L2 for every CTA of the
    // launch), and leave the factor in shared memory.
    float rs0 = 1.f, rs1 = 1.f;
    if (p.ssq_in) {
      float* row_rs = reinterpret_cast<float*>(sm + L::RS_OFF);
      const int t = (int)threadIdx.x - 64, r = t >> 1;
      float s = 0.f;
      if (r < p.m) {
        const float* src = p.ssq_in + (size_t)r * p.nt_in;
        if ((p.nt_in & 3) == 0) {
#pragma unroll 4
          for (int i = t & 1; i < p.nt_in / 4; i += 2) {
            const float4 x = __ldcg(reinterpret_cast<const float4*>(src) + i);
            s += (x.x + x.y) + (x.z + x.w);
          }
        } else {
          for (int i = t & 1; i < p.nt_in; i += 2) s += __ldcg(src + i);
        }
      }
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      if ((t & 1) == 0) row_rs[r] = rsqrtf(s * p.inv_h + p.eps) * (A8 && r < p.m ? __ldcg(p.x_scale + r) : 1.f);
      asm volatile("bar.sync 1, 128;" ::: "memory");
      rs0 = row_rs[lane];
      rs1 = row_rs[lane + 32];
    }
    for (int it = blockIdx.x; it < n_items; it += gridDim.x, ++local) {
      const int tile = it % total_tiles, split = it / total_tiles;
      const int acc = local % NACC;
      const uint32_t acc_phase = (uint32_t)(local / NACC) & 1u;
      ok = ok && mbar_wait(tfull_bar(acc), acc_phase, abort_flag);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float v[M_PAD];
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * ACC_COLS);
#pragma unroll
      for (int c = 0; c < M_PAD; c += 16) tmem_ld16(taddr + c, v + c);
      if (X3) {                    // x = p0 + p1 / 4 + p2 / 128
#pragma unroll
        for (int c = 0; c < M_PAD; c += 16) {
          float b1[16], b2[16];
          tmem_ld16(taddr + M_PAD + c, b1);
          tmem_ld16(taddr + 2 * M_PAD + c, b2);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int i = 0; i < 16; ++i) v[c + i] += fmaf(b2[i], 0.0078125f, b1[i] * 0.25f);
        }
      } else if (p.has_lo) {      // the low-order plane's product sits M_PAD columns further on
#pragma unroll
        for (int c = 0; c < M_PAD; c += 16) {
          float lo[16];
          tmem_ld16(taddr + M_PAD + c, lo);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int i = 0; i < 16; ++i) v[c + i] += lo[i];
        }
      }
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0 && ok) mbar_arrive(tempty_bar(acc));

      if (p.mode == TC_MODE_SWIGLU) {
        // Warps 0, 1 of the epilogue hold the gate values of features 32 pr + lane, warps 2, 3 the up values of the
        // same features.  Each warp of a pair finishes half of the rows: it hands the other half of its values
        // (scaled) to its partner through shared memory and takes the partner's values for its own rows.
        constexpr int HALF = M_PAD / 2;
        constexpr int ROUNDS = L::EX_ROUNDS;
        static_assert(HALF % ROUNDS == 0, "rows per round");
        constexpr int HR = HALF / ROUNDS;
        const int side = q >> 1, pr = q & 1;
        const int col = tile * 64 + pr * 32 + lane;
        const bool live = col < p.inter;
        const float sc = (live && p.scale[side]) ? p.scale[side][col] : 1.f;
        float* ex = reinterpret_cast<float*>(sm + L::EX_OFF) + pr * (2 * HR * 32);   // [side][HR rows][32 lanes]
#pragma unroll
        for (int r = 0; r < ROUNDS; ++r) {
          const uint32_t par = (uint32_t)(local * ROUNDS + r) & 1u;
#pragma unroll
          for (int b = 0; b < HR; ++b) {
            // the gate side finishes rows 0 .. HALF-1 and sends its values of rows HALF ..; the up side the reverse
            const int lo = r * HR + b, hi = HALF + r * HR + b;
            const float rs_lo = __shfl_sync(0xffffffffu, (lo < 32) ? rs0 : rs1, lo & 31);
            const float rs_hi = __shfl_sync(0xffffffffu, (hi < 32) ? rs0 : rs1, hi & 31);
            ex[(side * HR + b) * 32 + lane] = side ? v[lo] * sc * rs_lo : v[hi] * sc * rs_hi;
          }
          __syncwarp();
          if (lane == 0 && ok) mbar_arrive(exw_bar(pr));
          ok = ok && mbar_wait(exw_bar(pr), par, abort_flag);
          float am[HR];
#pragma unroll
          for (int b = 0; b < HR; ++b) {
            const int lo = r * HR + b, hi = HALF + r * HR + b;
            const float rs_lo = __shfl_sync(0xffffffffu, (lo < 32) ? rs0 : rs1, lo & 31);
            const float rs_hi = __shfl_sync(0xffffffffu, (hi < 32) ? rs0 : rs1, hi & 31);
            const float other = ex[((1 - side) * HR + b) * 32 + lane];
            const float mine = side ? v[hi] * sc * rs_hi : v[lo] * sc * rs_lo;
            const float g = side ? other : mine, u = side ? mine : other;
            const int row = side ? hi : lo;
            const float val = silu_mul(g, u);
            if (live && row < p.m) store_act(p.act, p.act_lo_off, (size_t)row * p.inter + col, val, p.act_fmt);
            if (A8) am[b] = (live && row < p.m) ? fabsf(__half2float(__ushort_as_half(f16_bits_sat(val)))) : 0.f;
          }
          if constexpr (A8) {
            // maxima of |act| as stored (f16) over this warp's 32 features, for whoever quantises the rows: non-negative values,
            // whose bit patterns order like integers (and the result does not depend on the order)
            const float mx = warp_reduce_transposed<true, HR>(am, lane);
            const int row = (side ? HALF : 0) + r * HR + lane;
            if (lane < HR && row < p.m && mx > 0.f) atomicMax(reinterpret_cast<int*>(p.amax_out) + row, __float_as_int(mx));
          }
          __syncwarp();
          if (lane == 0 && ok) mbar_arrive(exr_bar(pr));
          // the buffer may be rewritten once the partner has read it too
          ok = ok && mbar_wait(exr_bar(pr), par, abort_flag);
        }
      } else if (p.mode == TC_MODE_LOGITS) {
        const int n = tile * TC_BM + q * 32 + lane;          // vocabulary id held by this lane
        const bool in_range = n < p.n_out[0];
        const bool counted = in_range && n != p.mask_id;
        const float sc = (in_range && p.scale[0]) ? p.scale[0][n] : 1.f;
        // G rows at a time: their maxima and sums over the lanes are formed together (one row at a time, 15 shuffles each, made
        // this epilogue longer than the main loop at 64 rows: LM head of the 3B shape 160 us, 112 us now)
        constexpr int G = M_PAD % 32 == 0 ? 32 : 16;
#pragma unroll
        for (int b0 = 0; b0 < M_PAD; b0 += G) {
          if (b0 >= p.m) break;                               // uniform across the warp
          float w[G];
#pragma unroll
          for (int b = 0; b < G; ++b) {
            const float rs = __shfl_sync(0xffffffffu, (b0 + b < 32) ? rs0 : rs1, (b0 + b) & 31);
            const float l = v[b0 + b] * sc * rs;
            if (p.write_logits && in_range && b0 + b < p.m) p.y[(size_t)(b0 + b) * p.ldy + n] = l;
            v[b0 + b] = counted ? l : -INFINITY;
            w[b] = v[b0 + b];
          }
          const float mx = warp_reduce_transposed<true, G>(w, lane);         // of row b0 + lane mod G
          int first = 0;
#pragma unroll
          for (int b = 0; b < G; ++b) {
            const float m = __shfl_sync(0xffffffffu, mx, b);
            const unsigned at = __ballot_sync(0xffffffffu, v[b0 + b] == m);  // ids ascend with the lane: the lowest holds the argmax
            if ((lane & (G - 1)) == b) first = __ffs(at) - 1;
            w[b] = m > -INFINITY ? __expf(v[b0 + b] - m) : 0.f;
          }
          const float sum = warp_reduce_transposed<false, G>(w, lane);
          if (lane < G && b0 + lane < p.m)
            p.stats[(size_t)(tile * 4 + q) * p.m + b0 + lane] =
                make_float4(mx, sum, __int_as_float(mx > -INFINITY ? tile * TC_BM + q * 32 + first : 0x7fffffff), 0.f);
        }
      } else {
        int mi = 0;
        while (mi + 1 < p.n_mats && tile >= p.tile_begin[mi + 1]) ++mi;
        const int n = (tile - p.tile_begin[mi]) * TC_BM + q * 32 + lane;
        const bool in_range = n < p.n_out[mi];
        const int col = p.out_col[mi] + n;
        if (in_range) {
          float* dst = p.part + (size_t)split * p.m * p.ldp + col;
#pragma unroll
          for (int b = 0; b < M_PAD; ++b)
            if (b < p.m) dst[(size_t)b * p.ldp] = v[b];
        }
      }
    }
    if (!ok) {
      atomicCAS(p.status, 0, TC_ERR_EPILOGUE);
      linger();
    }
  }

  // ---- teardown: every thread arrives here, whatever happened ----
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
  if (threadIdx.x == 0) stamp_end(p.stamp);
}

// ================================================================================================
// host side
// ================================================================================================
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qr) == cudaSuccess &&
        qr == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)ptr;
  });
  return fn;
}

// Row-major [rows, cols] matrix, or `planes` > 0 of them plane_bytes apart as one 3-D tensor; box {64 columns, box_rows(, planes)}, zero
// OOB fill.  16-bit elements (TM_BF16, TM_F16): 128-byte swizzle (rows of the box are 128 bytes); e4m3 bytes: TM_E4M3 no swizzle (rows of
// 64 bytes, widened by the converter warps of the prompt path), TM_E4M3_128 a box of 128 columns with the 128-byte swizzle (the tile is an
// MMA operand as it lands).  A map is a function of these arguments alone: those made before are kept, at most 4096 of them.
static bool encode_tmap(CUtensorMap* tm, const void* ptr, int rows, int cols, int box_rows, int kind, int planes, size_t plane_bytes) {
  typedef std::tuple<const void*, int, int, int, int, int, size_t> Key;
  static std::map<Key, CUtensorMap> cache;
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  const bool fp8 = kind == TM_E4M3 || kind == TM_E4M3_128;
  const bool wide = kind == TM_E4M3_128;
  Key key(ptr, rows, cols, box_rows, kind, planes, plane_bytes);
  auto it = cache.find(key);
  if (it != cache.end()) { *tm = it->second; return true; }
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)cols * (fp8 ? 1 : 2), (cuuint64_t)plane_bytes};
  cuuint32_t box[3] = {(cuuint32_t)(wide ? 2 * TC_BK : TC_BK), (cuuint32_t)box_rows, (cuuint32_t)planes};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUtensorMapDataType dt = fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : (kind == TM_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16);
  CUresult r = fn(tm, dt, planes ? 3 : 2, const_cast<void*>(ptr), dims, strides,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, (fp8 && !wide) ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  if (cache.size() > 4096) cache.clear();
  cache[key] = *tm;
  return true;
}
bool make_tmap(CUtensorMap* tm, const void* ptr, int rows, int cols, int box_rows, int kind) {
  return encode_tmap(tm, ptr, rows, cols, box_rows, kind, 0, 0);
}
bool make_tmap_planes(CUtensorMap* tm, const void* ptr, int rows, int cols, int planes, size_t plane_bytes, int box_rows, int kind) {
  return encode_tmap(tm, ptr, rows, cols, box_rows, kind, planes, plane_bytes);
}

// (w1 nullable)
bool next_weights(NextWeights* n, const void* w0, const void* w1, int rows, int k, bool fp8, int step) {
  const void* w[2] = {w0, w1};
  n->mats = w1 ? 2 : 1;
  for (int i = 0; i < n->mats; ++i)
    if (!make_tmap(&n->tm[i], w[i], rows, k, 64, fp8 ? TM_E4M3_128 : TM_BF16)) return false;
  n->kb_elems = fp8 ? 2 * TC_BK : TC_BK;
  n->kblocks = ceil_div(k, n->kb_elems);
  n->step = step;
  n->row_blocks = ceil_div(rows, 64);
  n->units = n->row_blocks * ceil_div(ceil_div(n->kblocks, 2), step);
  return true;
}

// SM count of the current device (cached per device: one process may drive several GPUs)
int sm_count() {
  static int n[MAX_DEVICES] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return 148;
  if (!n[dev]) {
    int v = 0;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    n[dev] = v > 0 ? v : 148;
  }
  return n[dev];
}

static int pad_m(int m) { return m <= 16 ? 16 : (m <= 32 ? 32 : (m <= 48 ? 48 : 64)); }

// Split-K plan: enough (tile, split) items to occupy every SM about twice, each split at least 2
// k-blocks deep, never more splits than k-blocks.
static void tc_plan(int tiles, int kblocks, int* splits, int* kbps) {
  int s = (2 * sm_count()) / tiles;
  if (s < 1) s = 1;
  int max_s = kblocks / 2 > 0 ? kblocks / 2 : 1;
  if (s > max_s) s = max_s;
  if (s > 32) s = 32;
  int per = ceil_div(kblocks, s);
  *kbps = per;
  *splits = ceil_div(kblocks, per);
}

bool tc_linear_supported(int m, int n, int k, int dtype) {
  if (m < 1 || m > 64 || n < 1 || encode_fn() == nullptr) return false;
  if (dtype == DT_BF16) return k >= 8 && (k % 8) == 0;
  if (dtype == DT_FP8) return k >= 16 && (k % 16) == 0;     // byte rows must be 16-byte multiples for TMA
  return false;
}

size_t tc_workspace_bytes(int m, int ld, int tiles, int k) {
  int s, s8, kbps;       // (k-blocks of 64 elements, of 128 with fp8 weights)
  tc_plan(tiles, ceil_div(k, TC_BK), &s, &kbps);
  tc_plan(tiles, ceil_div(k, 2 * TC_BK), &s8, &kbps);
  return (size_t)(s > s8 ? s : s8) * m * ld * sizeof(float);
}

template <int M_PAD, int KIND>
static cudaError_t tc_launch_t(const TcParams& p, int grid, cudaStream_t st) {
  static bool attr_set[MAX_DEVICES] = {};
  cudaError_t e = ensure_dynamic_smem(gemm_tc_kernel<M_PAD, KIND>, TcSmem<M_PAD, KIND>::TOTAL, attr_set);
  if (e != cudaSuccess) return e;
  return launch_pdl(gemm_tc_kernel<M_PAD, KIND>, dim3(grid), dim3(TC_THREADS),
                    (size_t)TcSmem<M_PAD, KIND>::TOTAL, st, p);
}

template <int FP8>
static cudaError_t tc_launch_f(const TcParams& p, cudaStream_t st) {
  const int items = p.tile_begin[p.n_mats] * p.splits;
  const int grid = items < 2 * sm_count() ? items : 2 * sm_count();
  switch (pad_m(p.m)) {
    case 16: return tc_launch_t<16, FP8>(p, grid, st);
    case 32: return tc_launch_t<32, FP8>(p, grid, st);
    case 48: return tc_launch_t<48, FP8>(p, grid, st);
    default: return tc_launch_t<64, FP8>(p, grid, st);
  }
}

// A group of up to three bf16 matrices that share x and K, outputs side by side in one row of width ld.
//   mode PARTIAL: part[split][m][ld] (split-K sums left to the caller's reduce kernel); *splits_out tells how many
//   mode SWIGLU : act[m][inter] = silu(x wg^T * sg) * (x wu^T * su)  (w[0] = gate, w[1] = up; one split)

cudaError_t tc_group_launch(const TcGroup& g, const TcOut& o, cudaStream_t st) {
  TcParams p;
  memset(&p, 0, sizeof(p));
  const int mode = o.mode;
  const int mp = pad_m(g.m);
  const bool a8 = g.fp8 && g.a8;                  // rows as e4m3 codes
  const bool x3 = g.fp8 && !a8;                   // rows as e5m2 planes
  const int xkind = g.fp8 ? TM_E4M3_128 : TM_BF16;     // (bytes are bytes: e5m2 planes take the same map)
  if (a8 && mode == TC_MODE_LOGITS) return cudaErrorInvalidValue;
  if (a8 && mode == TC_MODE_SWIGLU && (!o.x_scale || !o.amax_out || !o.ssq_in)) return cudaErrorInvalidValue;
  if (!make_tmap(&p.tm_x, g.x, g.m, g.k, mp, xkind)) return cudaErrorInvalidValue;
  p.has_lo = (!g.fp8 && g.x_lo) ? 1 : 0;
  if ((x3 || p.has_lo) && !make_tmap(&p.tm_xl, g.x_lo, g.m, g.k, mp, xkind)) return cudaErrorInvalidValue;
  if (x3 && !make_tmap(&p.tm_x3, g.x_3, g.m, g.k, mp, xkind)) return cudaErrorInvalidValue;
  int tiles = 0, col = 0;
  for (int i = 0; i < g.n_mats; ++i) {
    if (!make_tmap(&p.tm_w[i], g.w[i], g.n[i], g.k, 64, g.fp8 ? TM_E4M3_128 : TM_BF16)) return cudaErrorInvalidValue;
    p.n_out[i] = g.n[i];
    p.tile_begin[i] = tiles;
    p.out_col[i] = col;
    p.scale[i] = g.scale[i];
    tiles += ceil_div(g.n[i], TC_BM);
    col += g.n[i];
  }
  p.n_mats = g.n_mats;
  p.kblocks = ceil_div(g.k, g.fp8 ? 2 * TC_BK : TC_BK);
  p.m = g.m;
  p.x_scale = o.x_scale; p.amax_out = o.amax_out;
  p.mode = mode;
  p.status = o.status;
  p.stamp = o.stamp;
  p.ssq_in = o.ssq_in; p.nt_in = o.nt_in; p.inv_h = o.hidden > 0 ? 1.f / (float)o.hidden : 0.f; p.eps = o.eps;
  if (mode == TC_MODE_SWIGLU) {
    tiles = ceil_div(g.n[0], 64);      // one combined list of 64-feature tiles (gate + up rows interleaved)
    p.n_mats = 1;
    p.tile_begin[0] = 0; p.tile_begin[1] = tiles;
    p.splits = 1; p.kb_per_split = p.kblocks;
    p.act = o.act; p.act_lo_off = o.act_lo_off; p.act_fmt = o.act_fmt; p.inter = g.n[0];
  } else {
    p.tile_begin[g.n_mats] = tiles;
    if (mode == TC_MODE_PARTIAL) tc_plan(tiles, p.kblocks, &p.splits, &p.kb_per_split);
    else { p.splits = 1; p.kb_per_split = p.kblocks; }
    p.part = o.part; p.ldp = o.ld; p.y = o.y; p.ldy = o.ld;
    p.stats = (float4*)o.stats; p.mask_id = o.mask_id; p.write_logits = o.write_logits;
    if (mode == TC_MODE_PARTIAL && (size_t)p.splits * g.m * o.ld * sizeof(float) > o.part_bytes) return cudaErrorInvalidValue;
    if (mode == TC_MODE_LOGITS && (g.n_mats != 1 || !o.stats)) return cudaErrorInvalidValue;
  }
  if (o.splits_out) *o.splits_out = p.splits;
  return a8 ? tc_launch_f<TC_KIND_A8>(p, st) : (g.fp8 ? tc_launch_f<TC_KIND_FP8>(p, st) : tc_launch_f<TC_KIND_BF16>(p, st));
}

}  // namespace fdk
