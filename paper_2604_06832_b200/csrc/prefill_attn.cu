// Causal GQA attention of the prompt path: row i (position L + i) reads keys 0 .. L + i.
//
// One CTA = two tiles of 128 consecutive rows of one query head.  S = Q K^T and O += P V run on the 5th-generation tensor
// cores (tcgen05.mma, 64 keys at a time) with S, P and O in tensor memory: P replaces S in place and is the A operand of
// the second product from there.  One softmax thread owns a row, so the online softmax needs no shuffles; O is rescaled
// only when a row's maximum has grown by more than 2^8, until then P is taken relative to the old reference (values up to
// 256, sums in fp32).  Each row tile has two score buffers, so the scores of the next keys are there when a softmax thread
// is done with its keys (one buffer of 128 keys: 97 us instead of 96 for 4096 rows of the 3B shape).  Bound by the
// exponentials, 16 per clock and SM.
// V stays as it lies in the cache ([key][dim], an MN-major operand).  Keys are not split and the normalised result is written directly as
// the O projection's input: 1024 rows of the 3B shape are 128 CTAs, one per SM (CTAs with the most keys come first).  A short turn
// is few CTAs (200 rows: 32), each of which walks all keys at 0.8 us per 64, so behind a long cache such turns take the decode
// path (takes_prompt_path).
// Every mbarrier wait is bounded as in gemm_tc.cu.
#include "attn_plan.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace fdk {

constexpr int PA_THREADS = 384;     // warp 0 TMA producer, warp 1 MMA issuer, warps 4..7 / 8..11 softmax of row tile 0 / 1
constexpr int PA_KEYS = 128;        // keys of a K / V tile in shared memory
constexpr int PA_STEP = 64;         // keys of one score buffer

template <int D>
struct PaSmem {
  static constexpr int TILE_BYTES = 128 * D * 2;        // a Q, K or V tile: D / 64 blocks of [128 rows][128 bytes], swizzled
  static constexpr int K_OFF = 2 * TILE_BYTES, V_OFF = K_OFF + 2 * TILE_BYTES;
  static constexpr int BAR_OFF = V_OFF + 2 * TILE_BYTES;
  static constexpr int TOTAL = BAR_OFF + 256 + 1024;
};

struct PaParams {
  CUtensorMap tm_q;           // [n, Hq * D], box {64, 128}
  CUtensorMap tm_k, tm_v;     // [Hkv * max_seq, D] planes, box {64, 128}
  void* out; size_t lo_off; int fmt;
  int n, L, max_seq, hq, hkv, rows;      // rows per CTA: 256 (both row tiles) or 128 (the first only)
  int* status;
  KStamp* stamp;
};

template <int D, typename E>
__global__ void __launch_bounds__(PA_THREADS, 1) prefill_attn_kernel(const __grid_constant__ PaParams p) {
  using S = PaSmem<D>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* sm = smem_raw + (base - raw);
  const uint32_t bar0 = base + S::BAR_OFF;
  const uint32_t q_full = bar0;
  auto k_full = [&](int s) { return bar0 + 8u + 8u * s; };
  auto k_empty = [&](int s) { return bar0 + 24u + 8u * s; };
  auto v_full = [&](int s) { return bar0 + 40u + 8u * s; };
  auto v_empty = [&](int s) { return bar0 + 56u + 8u * s; };
  auto s_full = [&](int q, int t) { return bar0 + 72u + 16u * q + 8u * (t & 1); };      // per score buffer
  auto p_full = [&](int q, int t) { return bar0 + 104u + 16u * q + 8u * (t & 1); };
  auto o_done = [&](int q) { return bar0 + 136u + 8u * q; };                            // a step's P V is complete
  auto o_full = [&](int q) { return bar0 + 152u + 8u * q; };                            // the last one is
  const uint32_t mma_done = bar0 + 176u;
  volatile uint32_t* tmem_slot = (volatile uint32_t*)(sm + S::BAR_OFF + 168);
  volatile int* abort_flag = (volatile int*)(sm + S::BAR_OFF + 172);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    stamp_start(p.stamp);
    mbar_init(q_full, 1); mbar_init(mma_done, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(k_full(i), 1); mbar_init(k_empty(i), 1); mbar_init(v_full(i), 1); mbar_init(v_empty(i), 1);
      for (int t = 0; t < 2; ++t) { mbar_init(s_full(i, t), 1); mbar_init(p_full(i, t), 4); }
      mbar_init(o_done(i), 1); mbar_init(o_full(i), 1);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;            // columns: score buffers (S, then P) of row tile q at 128 q and 128 q + 64, O at 256 + 128 q
  pdl_trigger();            // (holding its tensor memory: see gemm_tc.cu)
  pdl_wait();
  if (tid == 0) stamp_released(p.stamp);

  const int head = blockIdx.x, hk = head / (p.hq / p.hkv);
  const int i0 = (int)(gridDim.y - 1 - blockIdx.y) * p.rows;
  // steps of the two row tiles: up to the last row's own position (a row tile past the end of the prompt: none)
  const int rows0 = min(128, p.n - i0), rows1 = p.rows == 256 ? min(128, p.n - i0 - 128) : 0;
  const int n0 = (p.L + i0 + rows0 + PA_STEP - 1) / PA_STEP;
  const int n1 = rows1 > 0 ? (p.L + i0 + 128 + rows1 + PA_STEP - 1) / PA_STEP : 0;
  const int ns = max(n0, n1), nt = (ns + 1) / 2;

  if (warp == 0) {
    if (lane == 0) {
      const bool issue = may_issue(p.status, abort_flag);
      bool ok = issue;
      uint32_t k_armed = 0, v_armed = 0, k_par = 0, v_par = 0;
      if (ok) {
        mbar_expect_tx(q_full, 2 * S::TILE_BYTES);
        for (int q = 0; q < 2; ++q)
          for (int b = 0; b < D / 64; ++b)
            tma_load_2d_plain(base + q * S::TILE_BYTES + b * 16384, &p.tm_q, q_full, head * D + b * 64, i0 + q * 128);
      }
      for (int j = 0; j < nt && ok; ++j) {
        const int s = j & 1;
        const uint32_t ph = (uint32_t)(j >> 1) & 1u;
        const int row = hk * p.max_seq + j * PA_KEYS;
        if (!mbar_wait(k_empty(s), ph ^ 1u, abort_flag)) { ok = false; break; }
        mbar_expect_tx(k_full(s), S::TILE_BYTES);
        k_armed |= 1u << s; k_par = (k_par & ~(1u << s)) | (ph << s);
        for (int b = 0; b < D / 64; ++b) tma_load_2d_plain(base + S::K_OFF + s * S::TILE_BYTES + b * 16384, &p.tm_k, k_full(s), b * 64, row);
        if (!mbar_wait(v_empty(s), ph ^ 1u, abort_flag)) { ok = false; break; }
        mbar_expect_tx(v_full(s), S::TILE_BYTES);
        v_armed |= 1u << s; v_par = (v_par & ~(1u << s)) | (ph << s);
        for (int b = 0; b < D / 64; ++b) tma_load_2d_plain(base + S::V_OFF + s * S::TILE_BYTES + b * 16384, &p.tm_v, v_full(s), b * 64, row);
      }
      if (!ok && p.status) atomicCAS(p.status, 0, ST_ATTENTION);
      // no copy stays in flight, whether its reader has waited for it or has given up
      if (issue) mbar_drain(q_full, 0);
      for (int s = 0; s < 2; ++s) {
        if (k_armed & (1u << s)) mbar_drain(k_full(s), (k_par >> s) & 1u);
        if (v_armed & (1u << s)) mbar_drain(v_full(s), (v_par >> s) & 1u);
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {      // one thread issues everything: every election costs what several MMAs do (see gemm_gu.cu)
      constexpr bool F16 = sizeof(E) == 2 && !__is_same(E, bf16);
      const uint32_t id_s = F16 ? umma_idesc_f16(PA_STEP) : umma_idesc_bf16(PA_STEP);
      const uint32_t id_o = (F16 ? umma_idesc_f16(D) : umma_idesc_bf16(D)) | (1u << 16);      // (V: MN-major)
      bool ok = mbar_wait(q_full, 0, abort_flag);
      auto score = [&](int q, int t) {
        const uint32_t qa = base + q * S::TILE_BYTES, ka = base + S::K_OFF + ((t >> 1) & 1) * S::TILE_BYTES + (t & 1) * (PA_STEP * 128);
        if (ok) {
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk)
          umma_bf16(tmem + q * 128 + (t & 1) * PA_STEP, umma_desc_sw128(qa + (kk >> 2) * 16384) + 2u * (kk & 3),
                    umma_desc_sw128(ka + (kk >> 2) * 16384) + 2u * (kk & 3), id_s, kk > 0 ? 1u : 0u);
        umma_commit(s_full(q, t));
        }
      };
      auto value = [&](int q, int t) {
        ok = ok && mbar_wait(p_full(q, t), (uint32_t)(t >> 1) & 1u, abort_flag);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t vd = umma_desc_sw128_mn(base + S::V_OFF + ((t >> 1) & 1) * S::TILE_BYTES + (t & 1) * (PA_STEP * 128), 16384);
        if (ok) {
#pragma unroll
        for (int kk = 0; kk < PA_STEP / 16; ++kk)
          umma_f16_ta(tmem + 256 + q * 128, tmem + q * 128 + (t & 1) * PA_STEP + kk * 8, vd + (uint64_t)(kk * 128), id_o, (t > 0 || kk > 0) ? 1u : 0u);
        umma_commit(o_done(q));
        if (t + 1 == (q ? n1 : n0)) umma_commit(o_full(q));
        }
      };
      // the scores of step t for both row tiles; the K tile is free after its second half
      auto scores = [&](int q, int t) {
        if (t >= ns) return;
        if (q == 0 && (t & 1) == 0) {
          ok = ok && mbar_wait(k_full((t >> 1) & 1), (uint32_t)(t >> 2) & 1u, abort_flag);
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        if (t < (q ? n1 : n0)) score(q, t);
        if (q == 1 && ((t & 1) || t + 1 == ns)) { if (ok) umma_commit(k_empty((t >> 1) & 1)); }
      };
      for (int t = 0; t < 2; ++t) { scores(0, t); scores(1, t); }
      for (int t = 0; t < ns; ++t) {
        if ((t & 1) == 0) ok = ok && mbar_wait(v_full((t >> 1) & 1), (uint32_t)(t >> 2) & 1u, abort_flag);
        if (t < n0) value(0, t);
        scores(0, t + 2);
        if (t < n1) value(1, t);
        if ((t & 1) || t + 1 == ns) { if (ok) umma_commit(v_empty((t >> 1) & 1)); }
        scores(1, t + 2);
      }
      if (!ok && p.status) atomicCAS(p.status, 0, ST_ATTENTION);
      umma_commit(mma_done);      // no MMA outlives the tiles and the tensor memory that it uses, whoever gives up
      mbar_drain(mma_done, 0);
    }
    __syncwarp();
  } else if (warp >= 4) {
    const int q = (warp - 4) >> 2, wq = warp & 3;
    const int nq = q ? n1 : n0;
    const int i = i0 + q * 128 + wq * 32 + lane;              // this thread's row
    const int lim = p.L + min(i, p.n - 1) + 1;                // keys that it reads
    const int lim_first = p.L + i0 + q * 128 + wq * 32 + 1;   // keys that every row of the warp reads
    const int key_end = p.L + p.n;                            // (keys beyond this tile but before it are other rows' own)
    const uint32_t ts = tmem + ((uint32_t)(wq * 32) << 16) + q * 128, to = ts + 256;
    const float sl2 = rsqrtf((float)D) * LOG2E;               // scores in the log2 domain
    float m_ref = -INFINITY, l = 0.f;
    bool ok = true;
    for (int t = 0; t < nq; ++t) {
      ok = ok && mbar_wait(s_full(q, t), (uint32_t)(t >> 1) & 1u, abort_flag);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t tb = ts + (t & 1) * PA_STEP;
      float s[PA_STEP];
      tmem_ld32(tb, s);
      tmem_ld32(tb + 32, s + 32);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      const int j0 = t * PA_STEP;
      if (j0 + PA_STEP > lim_first) {                         // the diagonal (uniform over the warp)
#pragma unroll
        for (int c = 0; c < PA_STEP; ++c)
          if (j0 + c >= lim) s[c] = -INFINITY;
      }
      const float m = row_max64(s) * sl2;
      const bool grow = m > m_ref + 8.f;                      // (always in the first step: every row reads key 0)
      if (t > 0 && __any_sync(0xffffffffu, grow)) {
        ok = ok && mbar_wait(o_done(q), (uint32_t)(t - 1) & 1u, abort_flag);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const float f = grow ? ex2(m_ref - m) : 1.f;
        scale_acc<D>(to, f);
        l *= f;
      }
      if (grow) m_ref = m;
      l += exp_pack64<E>(s, sl2, m_ref, tb);
      if (j0 + PA_STEP > key_end) {
        // V rows past the last key hold whatever the cache holds there, and 0 x NaN would poison the product: cleared by
        // both row tiles (the same zeros)
        ok = ok && mbar_wait(v_full((t >> 1) & 1), (uint32_t)(t >> 2) & 1u, abort_flag);
        const int first = key_end - j0;
        for (int v = wq * 32 + lane; ok && v < (PA_STEP - first) * (D / 8); v += 128) {
          const int r = (t & 1) * PA_STEP + first + v / (D / 8), c = v % (D / 8);
          const uint32_t a = base + S::V_OFF + ((t >> 1) & 1) * S::TILE_BYTES + (c >> 3) * 16384 + r * 128 + (((c & 7) ^ (r & 7)) << 4);
          asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(a), "r"(0u) : "memory");
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0 && ok) mbar_arrive(p_full(q, t));
    }
    if (nq > 0) {
      ok = ok && mbar_wait(o_full(q), 0, abort_flag);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const float inv = 1.f / l;
      const size_t idx = ((size_t)i * p.hq + head) * D;
#pragma unroll 1
      for (int c = 0; c < D; c += 32) {
        float o[32];
        __syncwarp();
        tmem_ld32(to + c, o);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (ok && i < p.n) {
#pragma unroll
          for (int k = 0; k < 32; k += 4)
            store_act4(p.out, p.lo_off, idx + c + k, make_float4(o[k] * inv, o[k + 1] * inv, o[k + 2] * inv, o[k + 3] * inv), p.fmt);
        }
      }
    }
    if (!ok && p.status) atomicCAS(p.status, 0, ST_ATTENTION);
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();     // the producer's copies have all landed before any thread leaves
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
  if (tid == 0) stamp_end(p.stamp);
}

template <int D, typename E>
static cudaError_t pa_launch_t(const PaParams& p, cudaStream_t st) {
  using S = PaSmem<D>;
  static bool attr_set[MAX_DEVICES] = {};
  cudaError_t e = ensure_dynamic_smem(prefill_attn_kernel<D, E>, S::TOTAL, attr_set);
  if (e != cudaSuccess) return e;
  return launch_pdl(prefill_attn_kernel<D, E>, dim3(p.hq, ceil_div(p.n, p.rows)), dim3(PA_THREADS), (size_t)S::TOTAL, st, p);
}

cudaError_t launch_prefill_attention(const AttnArgs& a, cudaStream_t st) {
  PaParams p;
  memset(&p, 0, sizeof(p));
  const int kind = a.kv_type == KV_F16 ? TM_F16 : TM_BF16;
  if (!make_tmap(&p.tm_q, a.q, a.n, a.hq * a.d, 128, kind) || !make_tmap(&p.tm_k, a.kc, a.hkv * a.max_seq, a.d, PA_KEYS, kind) ||
      !make_tmap(&p.tm_v, a.vc, a.hkv * a.max_seq, a.d, PA_KEYS, kind))
    return cudaErrorInvalidValue;
  // Two row tiles per CTA share the K / V loads and keep the exponentials going; where CTAs of two do not even fill the SMs,
  // twice as many of one (1024 rows of the 3B shape 35 -> 25 us, 2048 rows 53 -> 43; 4096 rows 99 against 122).
  p.rows = a.hq * ceil_div(a.n, 256) <= sm_count() ? 128 : 256;
  p.out = a.out; p.lo_off = a.out_lo_off; p.fmt = a.out_fmt;
  p.n = a.n; p.L = a.cache_len; p.max_seq = a.max_seq; p.hq = a.hq; p.hkv = a.hkv; p.status = a.status; p.stamp = a.stamp;
  if (a.kv_type == KV_F16) return a.d == 128 ? pa_launch_t<128, __half>(p, st) : pa_launch_t<64, __half>(p, st);
  return a.d == 128 ? pa_launch_t<128, bf16>(p, st) : pa_launch_t<64, bf16>(p, st);
}

}  // namespace fdk
