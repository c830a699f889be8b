// Split-KV, block-masked GQA attention of the decode path (Sec. 3.3 masks; Alg. 1 draft / verify).
//
// One CTA = (KV head, group of query heads that share it, chunk of keys).  Its rows, at most 128, are the block's n rows of
// each of its query heads.  S = Q K^T and O += P V run on the 5th-generation tensor cores with S, P and O in tensor memory,
// as in the prompt path's kernel (prefill_attn.cu): one softmax thread owns a row, P replaces S in place, O is rescaled only
// when a row's maximum has grown by more than 2^8.  Here the two softmax warpgroups share the rows and take alternate
// 64-key steps (every 128-key tile is one step of each), with accumulators of their own that are added at the end: a short
// chunk is one step deep however it is cut.  K and V tiles are fetched by one producer warp with 2-D TMA loads; tiles that
// lie wholly in the committed cache are requested before the wait for the predecessor kernel.  Each CTA leaves an
// unnormalised partial (O, maximum, sum) and a small second kernel merges the chunks.  The in-block mask is applied by key
// index: denoise rows see all L + n keys, commit / prefill rows see keys <= L + i, or the caller gives bit masks.
// What bounds it is the chain through one CTA: rows to shared memory 1.5 us, S, softmax, P V, store (with mma.sync on 64-row CTAs: 13.4 us a layer at 8224 keys and 32 rows, 8.1 now; 5.5 and 5.3 at 2052 keys and 4 rows).
// Every mbarrier wait is bounded; a wait that gives up records ST_ATTENTION in the status word and the CTA drains its
// copies in flight and returns.
#include "attn_plan.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace fdk {

constexpr int AT_THREADS = 384;     // warp 0 TMA producer, warp 1 MMA issuer, warps 4..7 / 8..11 softmax of even / odd steps
constexpr int AT_ROWS = 128, AT_STEP = 64;

template <int D>
struct AtSmem {
  static constexpr int STAGES = 3;
  static constexpr int TILE_BYTES = 128 * D * 2;             // a Q, K or V tile: D / 64 blocks of [128 rows][128 bytes], swizzled
  static constexpr int KV_OFF = TILE_BYTES;                  // stage: K, then V
  static constexpr int BAR_OFF = KV_OFF + STAGES * 2 * TILE_BYTES;
  static constexpr int TOTAL = BAR_OFF + 256 + 1024;         // + alignment slack
  // the K / V ring doubles as the exchange of the epilogue: the rows' (m, l) of both warpgroups, 2 KB per warp to turn
  static constexpr int ML_OFF = KV_OFF, TURN_OFF = KV_OFF + 2048;
};

struct AttnParams {
  CUtensorMap tm_k, tm_v;     // [Hkv * max_seq, D] views of the layer's K and V planes, box {64, 128}
  const void* q;              // [n, Hq, D]
  float* part_o;              // [Hq][n][chunks][D]
  float2* part_ml;            // [Hq][n][chunks]
  int n, L, max_seq, hq, hkv, qh, chunk_keys, n_chunks, causal;
  const int* len_ptr;         // nullable: the cache length is read from device memory and the chunking derived from it
  const unsigned long long* row_mask;   // nullable: bit r' of word r = row r reads row r' of this forward (AttnArgs::row_mask)
  int* status;                // nullable: status words (see TcOut::status)
  KStamp* stamp;
  NextWeights next;
};

template <int D, typename E>
__global__ void __launch_bounds__(AT_THREADS, 1) attn_tc_kernel(const __grid_constant__ AttnParams p) {
  using S = AtSmem<D>;
  constexpr int CH = D / 8;                 // 16-byte chunks per row
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* sm = smem_raw + (base - raw);
  const uint32_t bar0 = base + S::BAR_OFF;
  const uint32_t q_full = bar0;
  auto k_full = [&](int s) { return bar0 + 8u + 8u * s; };
  auto v_full = [&](int s) { return bar0 + 32u + 8u * s; };
  auto kv_empty = [&](int s) { return bar0 + 56u + 8u * s; };
  auto s_full = [&](int w) { return bar0 + 80u + 8u * w; };
  auto p_full = [&](int w) { return bar0 + 96u + 8u * w; };
  auto o_full = [&](int w) { return bar0 + 112u + 8u * w; };     // the last P V of a warpgroup's steps is complete
  const uint32_t mma_done = bar0 + 136u;                         // every MMA is complete (after an abort)
  volatile uint32_t* tmem_slot = (volatile uint32_t*)(sm + S::BAR_OFF + 128);
  volatile int* abort_flag = (volatile int*)(sm + S::BAR_OFF + 132);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  int L = p.L, chunk_keys = p.chunk_keys, n_chunks = p.n_chunks;
  if (p.len_ptr) {   // the length word is written before the forward starts, not by a predecessor kernel
    L = *p.len_ptr;
    attn_chunking(L + p.n, (int)gridDim.x, &chunk_keys, &n_chunks);
  }
  const int n = p.n, hq = p.hq, hkv = p.hkv, qh = p.qh;
  const int chunk = blockIdx.x, grp = blockIdx.y, hk = blockIdx.z;
  const int cta = chunk + gridDim.x * (grp + gridDim.y * hk), ctas = gridDim.x * gridDim.y * gridDim.z;
  if (chunk >= n_chunks) {
    pdl_trigger();
    if (tid == 0) ask_for_next(p.next, cta, ctas);
    pdl_wait();
    return;
  }
  if (tid == 0) {
    stamp_start(p.stamp);
    mbar_init(q_full, 8); mbar_init(mma_done, 1);
    for (int i = 0; i < S::STAGES; ++i) { mbar_init(k_full(i), 1); mbar_init(v_full(i), 1); mbar_init(kv_empty(i), 1); }
    for (int w = 0; w < 2; ++w) { mbar_init(s_full(w), 1); mbar_init(p_full(w), 4); mbar_init(o_full(w), 1); }
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
  const uint32_t tmem = *tmem_slot;     // columns: S (then P) of warpgroup w at 64 w, O at 256 + 128 w
  pdl_trigger();                        // (holding its tensor memory: see gemm_tc.cu)

  const int G = hq / hkv;
  const int head0 = hk * G + grp * qh;                 // first query head of this CTA
  const int m_valid = min(qh, G - grp * qh) * n;
  const int key_begin = chunk * chunk_keys;
  const int key_end = min(L + n, key_begin + chunk_keys);
  const int n_tiles = (key_end - key_begin + AT_KEYS - 1) / AT_KEYS;
  // steps of warpgroup w: the w-th half of every tile that begins before the chunk's end
  const int steps0 = n_tiles, steps1 = key_begin + (n_tiles - 1) * AT_KEYS + AT_STEP < key_end ? n_tiles : n_tiles - 1;

  if (warp == 0) {
    if (lane == 0) {
      const uint64_t pol = policy_evict_last();     // the cache is read again by the other head groups and by the next step
      bool ok = may_issue(p.status, abort_flag), waited = false;
      uint32_t armed = 0, parity = 0;
      for (int t = 0; t < n_tiles && ok; ++t) {
        const int s = t % S::STAGES;
        const uint32_t ph = (uint32_t)(t / S::STAGES) & 1u;
        const int j0 = key_begin + t * AT_KEYS;
        // rows >= L are written by the predecessor kernel (the block's own K / V)
        if (!waited && j0 + AT_KEYS > L) { pdl_wait(); waited = true; }
        if (!mbar_wait(kv_empty(s), ph ^ 1u, abort_flag)) { ok = false; break; }
        armed |= 1u << s; parity = (parity & ~(1u << s)) | (ph << s);
        const uint32_t dst = base + S::KV_OFF + s * 2 * S::TILE_BYTES;
        const int row = hk * p.max_seq + j0;
        mbar_expect_tx(k_full(s), S::TILE_BYTES);
#pragma unroll
        for (int b = 0; b < D / 64; ++b) tma_load_2d(dst + b * 16384, &p.tm_k, k_full(s), b * 64, row, pol);
        mbar_expect_tx(v_full(s), S::TILE_BYTES);
#pragma unroll
        for (int b = 0; b < D / 64; ++b) tma_load_2d(dst + S::TILE_BYTES + b * 16384, &p.tm_v, v_full(s), b * 64, row, pol);
      }
      if (!waited) pdl_wait();
      if (!ok && p.status) atomicCAS(p.status, 0, ST_ATTENTION);
      if (*abort_flag)      // (see linger)
        for (int s = 0; s < S::STAGES; ++s)
          if (armed & (1u << s)) {
            mbar_drain(k_full(s), (parity >> s) & 1u);
            mbar_drain(v_full(s), (parity >> s) & 1u);
          }
    }
  } else if (warp == 1) {
    constexpr bool F16 = !__is_same(E, bf16);
    const uint32_t id_s = F16 ? umma_idesc_f16(AT_STEP) : umma_idesc_bf16(AT_STEP);
    const uint32_t id_o = (F16 ? umma_idesc_f16(D) : umma_idesc_bf16(D)) | (1u << 16);      // (V: MN-major)
    if (elect_one()) {      // one thread issues everything: every election costs what several MMAs do (see gemm_gu.cu)
      bool ok = mbar_wait(q_full, 0, abort_flag);
      auto score = [&](int w, int t) {
        if (t >= (w ? steps1 : steps0)) return;
        const int s = t % S::STAGES;
        ok = ok && mbar_wait(k_full(s), (uint32_t)(t / S::STAGES) & 1u, abort_flag);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t ka = base + S::KV_OFF + s * 2 * S::TILE_BYTES + w * (AT_STEP * 128);
        if (ok) {
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk)
            umma_bf16(tmem + w * AT_STEP, umma_desc_sw128(base + (kk >> 2) * 16384) + 2u * (kk & 3), umma_desc_sw128(ka + (kk >> 2) * 16384) + 2u * (kk & 3),
                      id_s, kk > 0 ? 1u : 0u);
          umma_commit(s_full(w));
        }
      };
      auto value = [&](int w, int t) {
        const int steps = w ? steps1 : steps0;
        if (t >= steps) return;
        const int s = t % S::STAGES;
        ok = ok && mbar_wait(p_full(w), (uint32_t)t & 1u, abort_flag) && mbar_wait(v_full(s), (uint32_t)(t / S::STAGES) & 1u, abort_flag);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t vd = umma_desc_sw128_mn(base + S::KV_OFF + (s * 2 + 1) * S::TILE_BYTES + w * (AT_STEP * 128), 16384);
        if (ok) {
#pragma unroll
          for (int kk = 0; kk < AT_STEP / 16; ++kk)
            umma_f16_ta(tmem + 256 + w * 128, tmem + w * AT_STEP + kk * 8, vd + (uint64_t)(kk * 128), id_o, (t > 0 || kk > 0) ? 1u : 0u);
          if (t + 1 == steps) umma_commit(o_full(w));
        }
      };
      score(0, 0);
      score(1, 0);
      for (int t = 0; t < n_tiles; ++t) {
        value(0, t);
        score(0, t + 1);
        value(1, t);
        if (ok) umma_commit(kv_empty(t % S::STAGES));
        score(1, t + 1);
      }
      if (!ok && p.status) atomicCAS(p.status, 0, ST_ATTENTION);
      if (*abort_flag) {
        umma_commit(mma_done);
        mbar_drain(mma_done, 0);
        linger();
      }
    }
    __syncwarp();
  } else if (warp >= 4) {
    // Where this thread's pieces of Q come from and its rows of the result go is worked out before the wait: rows = heads x n,
    // row r -> head r / n, token r % n.
    const int wt = tid - 128;
    const int w = (warp - 4) >> 2, wq = warp & 3;
    constexpr int NQ = AT_ROWS * CH / 256, RS = 256 / CH;     // 16-byte pieces per thread, rows between them
    int q_off[NQ], out_row[4];
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const int r = wt / CH + i * RS;
      q_off[i] = r < m_valid ? ((r % n) * hq + head0 + r / n) * D + (wt % CH) * 8 : -1;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = wq * 32 + (lane >> 2) + 8 * i;
      out_row[i] = r < m_valid ? ((head0 + r / n) * n + r % n) * n_chunks + chunk : -1;
    }
    const int row = wq * 32 + lane;                           // this thread's row; the other warpgroup has it too
    const bool row_live = row < m_valid;
    const int tok = row % n, slot = ((head0 + row / n) * n + tok) * n_chunks + chunk;
    const int lim = row_live && !p.causal ? L + n : L + tok + 1;      // keys it may read
    const unsigned long long mask = p.row_mask ? p.row_mask[tok] : ~0ull;      // (set up before the chain)
    // stage Q: written by the predecessor kernel
    pdl_wait();
    if (wt == 0) stamp_released(p.stamp);
    const E* q = reinterpret_cast<const E*>(p.q);
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const int r = wt / CH + i * RS, c = wt % CH;
      cp_async16(base + (c >> 3) * 16384 + r * 128 + (((c & 7) ^ (r & 7)) << 4), q + max(q_off[i], 0), q_off[i] >= 0 ? 16 : 0);
    }
    cp_async_commit();
    const uint32_t ts = tmem + ((uint32_t)(wq * 32) << 16) + w * AT_STEP;
    const uint32_t to = tmem + ((uint32_t)(wq * 32) << 16) + 256;
    const float sl2 = rsqrtf((float)D) * LOG2E;               // scores in the log2 domain
    float m_ref = -INFINITY, l = 0.f;
    bool ok = true;
    const int steps = w ? steps1 : steps0;
    cp_async_wait<0>();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // generic writes -> the MMA's async-proxy reads
    __syncwarp();
    if (lane == 0) mbar_arrive(q_full);
    for (int t = 0; t < steps; ++t) {
      ok = ok && mbar_wait(s_full(w), (uint32_t)t & 1u, abort_flag);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float s[AT_STEP];
      tmem_ld32(ts, s);
      tmem_ld32(ts + 32, s + 32);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      const int j0 = key_begin + t * AT_KEYS + w * AT_STEP;
      if (j0 + AT_STEP > L) {               // keys of the forward's own rows (uniform)
        // bit c: this row reads key j0 + c
        unsigned long long vis = j0 <= L ? (mask << (L - j0)) | ((1ull << (L - j0)) - 1ull) : (j0 - L < 64 ? mask >> (j0 - L) : 0ull);
        if (lim - j0 < 64) vis &= lim > j0 ? (1ull << (lim - j0)) - 1ull : 0ull;
        const uint32_t v0 = (uint32_t)vis, v1 = (uint32_t)(vis >> 32);
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          if (!(v0 & (1u << c))) s[c] = -INFINITY;
          if (!(v1 & (1u << c))) s[32 + c] = -INFINITY;
        }
      }
      const float m = row_max64(s) * sl2;
      const bool grow = m > m_ref + 8.f;
      if (t > 0 && __any_sync(0xffffffffu, grow)) {
        // (s_full also says that this warpgroup's product of the step before is complete: O may be rewritten)
        const float f = grow ? ex2(m_ref - m) : 1.f;
        scale_acc<D>(to + w * 128, f);
        l *= f;
      }
      if (grow) m_ref = m;
      l += exp_pack64<E>(s, sl2, m_ref == -INFINITY ? 0.f : m_ref, ts);
      if (j0 + AT_STEP > key_end) {
        // V rows past the last key hold whatever the cache holds there, and 0 x NaN would poison the product
        const int sg = t % S::STAGES, first = max(0, key_end - j0);
        ok = ok && mbar_wait(v_full(sg), (uint32_t)(t / S::STAGES) & 1u, abort_flag);
        for (int v = wq * 32 + lane; ok && v < (AT_STEP - first) * CH; v += 128) {
          const int r = w * AT_STEP + first + v / CH, c = v % CH;
          const uint32_t a = base + S::KV_OFF + (sg * 2 + 1) * S::TILE_BYTES + (c >> 3) * 16384 + r * 128 + (((c & 7) ^ (r & 7)) << 4);
          asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(a), "r"(0u) : "memory");
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0 && ok) mbar_arrive(p_full(w));
    }
    for (int x = 0; x < 2; ++x)
      if ((x ? steps1 : steps0) > 0) ok = ok && mbar_wait(o_full(x), 0, abort_flag);
    // every load has been used up and every product is complete: the ring is free.  Each warpgroup stores half of the
    // columns of the sum of both accumulators.
    ok = named_barrier_and<256>(ok);
    if (ok) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float2* ml = reinterpret_cast<float2*>(sm + S::ML_OFF);
      ml[w * 128 + row] = make_float2(m_ref, l);
      asm volatile("bar.sync 1, 256;" ::: "memory");
      const float2 other = ml[(1 - w) * 128 + row];
      const float m = fmaxf(m_ref, other.x), ref = m == -INFINITY ? 0.f : m;
      const float fm = ex2(m_ref - ref), fo = ex2(other.x - ref);
      const float f0 = w ? fo : fm, f1 = w ? fm : fo;
      if (w == 0 && row_live) p.part_ml[slot] = make_float2(m, l * fm + other.y * fo);
      // rows of a turned block: lane / 4 + 8 i, four columns each.  (16 columns at a time: this code runs once, and half the
      // instructions are fetched in half the time)
      const uint32_t buf = base + S::TURN_OFF + (warp - 4) * 2048;
      const int lc = (lane & 3) * 4;
#pragma unroll 1
      for (int c = w * (D / 2); c < (w + 1) * (D / 2); c += 16) {
        float a[16], b[16];
        float4 o[4];
        __syncwarp();
        tmem_ld16(to + c, a);
        tmem_ld16(to + 128 + c, b);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (steps1 == 0) {       // (the second accumulator was never written and holds anything)
#pragma unroll
          for (int k = 0; k < 16; ++k) b[k] = 0.f;
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) a[k] = fmaf(a[k], f0, b[k] * f1);
        turn<16>(buf, lane, a, o);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (out_row[i] >= 0) *reinterpret_cast<float4*>(p.part_o + (size_t)out_row[i] * D + c + lc) = o[i];
      }
    } else {
      if (lane == 0 && p.status) atomicCAS(p.status, 0, ST_ATTENTION);
      linger();
    }
  } else {
    if (warp == 2 && lane == 0) ask_for_next(p.next, cta, ctas);
    pdl_wait();
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();     // nothing is in flight any more (see linger)
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
  if (tid == 0) stamp_end(p.stamp);
}

// Merge of the key chunks: out[i][head] = sum_c w_c O_c / sum_c w_c l_c, w_c = 2^(m_c - max_c m_c).  WPP warps per
// (row, head): warp w takes the chunks w, w + WPP, ..., CB of them in flight at once; with WPP = 4 warp 0 adds up the four.
// Four where that is at most four CTAs per SM (one warp per pair took 5.4 us a layer for the 33 chunks of 8224 keys and 32
// rows of the 3B shape, four about 3.5), one beyond (64 rows: 3.4 against 4.1).  Lane j owns D / 32 consecutive output
// features.  The result is stored as `fmt` (XF_*).
template <int D, int WPP>
__global__ void __launch_bounds__(128) attn_combine_kernel(const float* __restrict__ part_o, const float2* __restrict__ part_ml,
                                                             void* __restrict__ out, size_t lo_off, int fmt, int n, int hq, int n_chunks,
                                                             const int* __restrict__ len_ptr, int bound, float* __restrict__ amax_out,
                                                             KStamp* stamp) {
  constexpr int VPL = D / 32, CB = WPP == 4 ? 10 : 20;
  if (threadIdx.x == 0) stamp_start(stamp);
  pdl_trigger();
  if (len_ptr) {
    int ck;
    attn_chunking(*len_ptr + n, bound, &ck, &n_chunks);
  }
  __shared__ float s_m[4], s_l[4];
  __shared__ __align__(16) float s_o[4][D];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pair = WPP == 4 ? blockIdx.x : blockIdx.x * 4 + warp;
  const bool live = pair < n * hq;
  const int i = pair / hq, head = pair - i * hq;
  const size_t slot0 = ((size_t)head * n + i) * n_chunks;
  const float* src = part_o + slot0 * D + lane * VPL;
  pdl_wait();
  if (threadIdx.x == 0) stamp_released(stamp);
  float m = -INFINITY, l = 0.f, acc[VPL];
#pragma unroll
  for (int k = 0; k < VPL; ++k) acc[k] = 0.f;
  for (int c0 = WPP == 4 ? warp : 0; live && c0 < n_chunks; c0 += WPP * CB) {
    float2 ml[CB];
    float o[CB][VPL];
#pragma unroll
    for (int u = 0; u < CB; ++u) {
      const int c = c0 + WPP * u;
      ml[u] = make_float2(-INFINITY, 0.f);
      if (c < n_chunks) {
        ml[u] = __ldcg(&part_ml[slot0 + c]);
        if (VPL == 4) {
          const float4 x = __ldcg(reinterpret_cast<const float4*>(src + (size_t)c * D));
          o[u][0] = x.x; o[u][1] = x.y; o[u][VPL - 2] = x.z; o[u][VPL - 1] = x.w;
        } else {
          const float2 x = __ldcg(reinterpret_cast<const float2*>(src + (size_t)c * D));
          o[u][0] = x.x; o[u][VPL - 1] = x.y;
        }
      }
    }
    float mn = m;
#pragma unroll
    for (int u = 0; u < CB; ++u) mn = fmaxf(mn, ml[u].x);
    if (mn == -INFINITY) continue;                 // (nothing visible so far; uniform over the warp)
    const float keep = exp2f(m - mn);
    m = mn;
    l *= keep;
#pragma unroll
    for (int k = 0; k < VPL; ++k) acc[k] *= keep;
#pragma unroll
    for (int u = 0; u < CB; ++u) {
      if (ml[u].y != 0.f) {
        const float w = exp2f(ml[u].x - m);
        l = fmaf(w, ml[u].y, l);
#pragma unroll
        for (int k = 0; k < VPL; ++k) acc[k] = fmaf(w, o[u][k], acc[k]);
      }
    }
  }
  if (WPP == 4) {
    if (lane == 0) { s_m[warp] = m; s_l[warp] = l; }
#pragma unroll
    for (int k = 0; k < VPL; ++k) s_o[warp][lane * VPL + k] = acc[k];
    __syncthreads();
  }
  if (WPP == 4 ? warp == 0 : live) {
    if (WPP == 4) {
      m = fmaxf(fmaxf(s_m[0], s_m[1]), fmaxf(s_m[2], s_m[3]));
      l = 0.f;
#pragma unroll
      for (int k = 0; k < VPL; ++k) acc[k] = 0.f;
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const float f = exp2f(s_m[w] - m);
        l = fmaf(f, s_l[w], l);
#pragma unroll
        for (int k = 0; k < VPL; ++k) acc[k] = fmaf(f, s_o[w][lane * VPL + k], acc[k]);
      }
    }
    const float inv = 1.f / l;
    const size_t idx = ((size_t)i * hq + head) * D + lane * VPL;
    // (a caller's `out` may lie at any element: four of them in one store only where they are aligned)
    if (VPL == 4 && (reinterpret_cast<uintptr_t>(out) & 7) == 0) {
      store_act4(out, lo_off, idx, make_float4(acc[0] * inv, acc[1] * inv, acc[VPL - 2] * inv, acc[VPL - 1] * inv), fmt);
    } else {
#pragma unroll
      for (int k = 0; k < VPL; ++k) store_act(out, lo_off, idx + k, acc[k] * inv, fmt);
    }
    if (amax_out) {     // W8A8: the O projection quantises this row; its maximum as stored (f16) over this head
      float am = 0.f;
#pragma unroll
      for (int k = 0; k < VPL; ++k) am = fmaxf(am, fabsf(__half2float(__ushort_as_half(f16_bits_sat(acc[k] * inv)))));
      am = warp_max(am);
      if (lane == 0) amax_out[(size_t)i * hq + head] = am;
    }
    if (lane == 0 && warp == 0) stamp_end(stamp, true);
  }
}

// ---- host side -------------------------------------------------------------------------------------
// The chunk merge that follows either attention kernel.  grid_x: the chunk slots the partials were laid out for.
cudaError_t launch_attn_combine(const float* part_o, const float2* part_ml, const AttnArgs& a, int n_chunks, int grid_x,
                                KStamp* stamp, cudaStream_t st) {
  const int pairs = a.n * a.hq;
  const bool four = pairs <= 4 * sm_count();
  auto kern = a.d == 128 ? (four ? attn_combine_kernel<128, 4> : attn_combine_kernel<128, 1>) : (four ? attn_combine_kernel<64, 4> : attn_combine_kernel<64, 1>);
  const cudaError_t e = launch_pdl(kern, dim3(four ? pairs : (pairs + 3) / 4), dim3(128), 0, st, part_o, part_ml, a.out, a.out_lo_off, a.out_fmt,
                                   a.n, a.hq, n_chunks, a.len_ptr, grid_x, a.amax_out, stamp);
  return e != cudaSuccess ? e : cudaGetLastError();
}

struct AttnPlan { int qh, groups, chunk_keys, n_chunks, bound; };

// heads per CTA: the most query heads of one KV head whose n rows fit; chunks: one CTA per SM
static AttnPlan attn_plan(int n, int T, int hq, int hkv) {
  AttnPlan p;
  const int G = hq / hkv;
  p.qh = 1;
  for (int c = G; c >= 1; --c)
    if (c * n <= AT_ROWS) { p.qh = c; break; }
  p.groups = ceil_div(G, p.qh);
  p.bound = sm_count() / (hkv * p.groups);
  if (p.bound < 1) p.bound = 1;
  attn_chunking(T, p.bound, &p.chunk_keys, &p.n_chunks);
  return p;
}

size_t attention_tc_workspace_bytes(int n, int hq, int hkv, int d) {
  size_t worst = 0;
  for (int m = 1; m <= n; ++m) {
    const size_t slots = (size_t)hq * m * attn_plan(m, 1, hq, hkv).bound;
    if (slots > worst) worst = slots;
  }
  return worst * ((size_t)d * 4 + 8) + 256;
}

template <int D, typename E>
static cudaError_t attn_launch_t(const AttnArgs& a, const AttnPlan& pl, cudaStream_t st) {
  using S = AtSmem<D>;
  // with the length on the device the grid is sized for the most chunks any length can give
  int grid_x = pl.n_chunks;
  if (a.len_ptr) { grid_x = pl.bound; const int tmax = ceil_div(a.max_seq, AT_KEYS); if (grid_x > tmax) grid_x = tmax; }
  // One CTA per SM where next weights are asked for: those without a chunk take their share (with 24 CTAs of 16 rows the boxes of 34 MB were
  // still being issued when the attention was done: 766 us a step of 12 layers, 696 with 148)
  if (a.next_w[0]) grid_x = pl.bound;
  const size_t slots = (size_t)a.hq * a.n * grid_x;
  AttnParams p;
  memset(&p, 0, sizeof(p));
  const int kind = a.kv_type == KV_F16 ? TM_F16 : TM_BF16;
  if (!make_tmap(&p.tm_k, a.kc, a.hkv * a.max_seq, D, AT_KEYS, kind) || !make_tmap(&p.tm_v, a.vc, a.hkv * a.max_seq, D, AT_KEYS, kind))
    return cudaErrorInvalidValue;
  p.q = a.q;
  p.part_o = (float*)a.workspace;
  p.part_ml = (float2*)((char*)a.workspace + ((slots * D * 4 + 255) / 256) * 256);
  p.n = a.n; p.L = a.cache_len; p.max_seq = a.max_seq; p.hq = a.hq; p.hkv = a.hkv; p.qh = pl.qh;
  p.chunk_keys = pl.chunk_keys; p.n_chunks = pl.n_chunks; p.causal = a.row_mask ? 0 : a.causal; p.row_mask = a.row_mask; p.len_ptr = a.len_ptr; p.status = a.status; p.stamp = a.stamp;
  if (a.next_w[0] && !next_weights(&p.next, a.next_w[0], a.next_w[1], a.next_n, a.next_k, a.next_fp8 != 0, 3)) return cudaErrorInvalidValue;
  static bool attr_set[MAX_DEVICES] = {};
  cudaError_t e = ensure_dynamic_smem(attn_tc_kernel<D, E>, S::TOTAL, attr_set);
  if (e != cudaSuccess) return e;
  e = launch_pdl(attn_tc_kernel<D, E>, dim3(grid_x, pl.groups, a.hkv), dim3(AT_THREADS), (size_t)S::TOTAL, st, p);
  if (e != cudaSuccess) return e;
  return launch_attn_combine(p.part_o, p.part_ml, a, pl.n_chunks, grid_x, a.stamp ? a.stamp + 1 : nullptr, st);
}

int launch_attention_tc(const AttnArgs& a, cudaStream_t st, cudaError_t* err) {
  if (!a.workspace) { *err = cudaErrorInvalidValue; return -1; }
  const AttnPlan pl = attn_plan(a.n, a.cache_len + a.n, a.hq, a.hkv);
  if (a.kv_type == KV_F16) *err = (a.d == 128) ? attn_launch_t<128, __half>(a, pl, st) : attn_launch_t<64, __half>(a, pl, st);
  else *err = (a.d == 128) ? attn_launch_t<128, bf16>(a, pl, st) : attn_launch_t<64, bf16>(a, pl, st);
  return *err == cudaSuccess ? 2 : -1;
}

}  // namespace fdk
