// Causal GQA attention of the prompt path: row i (position L + i) reads keys 0 .. L + i.
//
// One CTA = 128 consecutive rows of one query head; eight compute warps of 16 rows each, one producer warp that fetches
// 64-key K and V tiles by 2-D TMA into a ring.  Hundreds of CTAs exist at any prompt length, so keys are not split and
// the normalised result is written directly as the O projection's input.  CTAs with the most keys come first.
// mma.sync m16n8k16, fp32 online softmax as in the decode kernel (attention.cu).
#include "attn_plan.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace fdk {

template <int D>
struct PaSmem {
  static constexpr int ROWS = 128, NW = ROWS / 16, THREADS = NW * 32 + 32;
  static constexpr int STAGES = D == 128 ? 4 : 8;
  static constexpr int Q_BYTES = ROWS * D * 2;
  static constexpr int TILE_BYTES = AT_KEYS * D * 2;
  static constexpr int STAGE_BYTES = 2 * TILE_BYTES;
  static constexpr int BAR_OFF = Q_BYTES + STAGES * STAGE_BYTES;
  static constexpr int TOTAL = BAR_OFF + 8 * (2 * STAGES) + 16 + 1024;
};

struct PaParams {
  CUtensorMap tm_k, tm_v;     // [Hkv * max_seq, D] planes, box {64, 64}
  const void* q;              // [n, Hq, D]
  void* out; size_t lo_off; int fmt;
  int n, L, max_seq, hq, hkv;
  int* status;
};

template <int D, typename E>
__global__ void __launch_bounds__(PaSmem<D>::THREADS, 1) prefill_attn_kernel(const __grid_constant__ PaParams p) {
  using S = PaSmem<D>;
  constexpr int CH = D / 8, NW = S::NW, NCT = NW * 32;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t sQ = (raw + 1023u) & ~1023u;
  uint8_t* sm = smem_raw + (sQ - raw);
  const uint32_t sKV = sQ + S::Q_BYTES, bar0 = sQ + S::BAR_OFF;
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (S::STAGES + s); };
  volatile int* abort_flag = (volatile int*)(sm + S::BAR_OFF + 8 * (2 * S::STAGES));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  pdl_trigger();
  if (tid == 0) {
    for (int s = 0; s < S::STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), NW); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  pdl_wait();
  const int head = blockIdx.x, hk = head / (p.hq / p.hkv);
  const int i0 = (int)(gridDim.y - 1 - blockIdx.y) * S::ROWS;
  const int rows = min(S::ROWS, p.n - i0);
  const int key_end = p.L + i0 + rows;                       // exclusive
  const int n_tiles = (key_end + AT_KEYS - 1) / AT_KEYS;

  if (warp == NW) {
    if (lane == 0) {
      const bool poisoned = p.status && *reinterpret_cast<const volatile int*>(p.status + 1) != 0;   // host-set test hook
      if (poisoned) *abort_flag = 1;
      bool ok = !poisoned;
      uint32_t armed = 0, armed_parity = 0;
      for (int t = 0; t < n_tiles && ok; ++t) {
        const int stage = t % S::STAGES;
        const uint32_t phase = (uint32_t)(t / S::STAGES) & 1u;
        if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag)) { ok = false; break; }
        mbar_expect_tx(full_bar(stage), S::STAGE_BYTES);
        armed |= 1u << stage;
        armed_parity = (armed_parity & ~(1u << stage)) | (phase << stage);
        const uint32_t dst = sKV + stage * S::STAGE_BYTES;
        const int row = hk * p.max_seq + t * AT_KEYS;
#pragma unroll
        for (int hd = 0; hd < D / 64; ++hd) {
          tma_load_2d_plain(dst + hd * (AT_KEYS * 128), &p.tm_k, full_bar(stage), hd * 64, row);
          tma_load_2d_plain(dst + S::TILE_BYTES + hd * (AT_KEYS * 128), &p.tm_v, full_bar(stage), hd * 64, row);
        }
      }
      if (!ok) {
        if (p.status) atomicCAS(p.status, 0, ST_ATTENTION);
        for (int s = 0; s < S::STAGES; ++s) {
          if (!(armed & (1u << s))) continue;
          const uint32_t par = (armed_parity >> s) & 1u;
          const long long t0 = clock64();
          while (!mbar_try_wait(full_bar(s), par) && clock64() - t0 < TC_TIMEOUT) {}
        }
      }
    }
  } else {
    const E* q = reinterpret_cast<const E*>(p.q);
    for (int v = tid; v < S::ROWS * CH; v += NCT) {
      const int r = v / CH, c = v % CH;
      const bool live = r < rows;
      cp_async16(sQ + swz_q<D>(r, c), live ? (const void*)(q + ((size_t)(i0 + r) * p.hq + head) * D + c * 8) : (const void*)q, live ? 16 : 0);
    }
    cp_async_commit();
    cp_async_wait<0>();
    asm volatile("bar.sync 1, %0;" ::"n"(NCT) : "memory");
    const int row0 = warp * 16, g = lane >> 2, tq = lane & 3;
    const int r_lo = row0 + g, r_hi = r_lo + 8;
    // last visible key (exclusive); a row past the end of the prompt sees none
    const int lim_lo = r_lo < rows ? p.L + i0 + r_lo + 1 : 0, lim_hi = r_hi < rows ? p.L + i0 + r_hi + 1 : 0;
    const int warp_first = p.L + i0 + row0 + 1;               // keys that every row of the warp sees
    const int warp_last = p.L + i0 + row0 + 16;               // keys beyond this are seen by none
    const float sl2 = rsqrtf((float)D) * LOG2E;
    uint32_t qf[D / 16][4];
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk)
      ldsm_x4(sQ + swz_q<D>(row0 + (lane & 15), kk * 2 + (lane >> 4)), qf[kk][0], qf[kk][1], qf[kk][2], qf[kk][3]);
    float o[D / 8][4];
#pragma unroll
    for (int i = 0; i < D / 8; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }
    float m_lo = -INFINITY, m_hi = -INFINITY, l_lo = 0.f, l_hi = 0.f;
    bool ok = true;
    for (int t = 0; t < n_tiles && ok; ++t) {
      const int stage = t % S::STAGES;
      const uint32_t phase = (uint32_t)(t / S::STAGES) & 1u;
      if (!mbar_wait(full_bar(stage), phase, abort_flag)) { ok = false; break; }
      const uint32_t kt = sKV + stage * S::STAGE_BYTES, vt = kt + S::TILE_BYTES;
      const int j0 = t * AT_KEYS;
      if (j0 + AT_KEYS > key_end) {
        // V rows past the last key hold whatever the cache holds there, and 0 x NaN would poison the product: every warp
        // clears them (the same zeros) before it reads any
        const int first = key_end - j0;
        for (int v = lane; v < (AT_KEYS - first) * CH; v += 32) {
          const int r = first + v / CH, c = v % CH;
          asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(vt + swz_kv(r, c)), "r"(0u) : "memory");
        }
        __syncwarp();
      }
      if (j0 < warp_last && row0 < rows) {
        float s[AT_KEYS / 8][4];
#pragma unroll
        for (int i = 0; i < AT_KEYS / 8; ++i) { s[i][0] = s[i][1] = s[i][2] = s[i][3] = 0.f; }
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
#pragma unroll
          for (int np = 0; np < AT_KEYS / 16; ++np) {
            uint32_t b0, b1, b2, b3;
            ldsm_x4(kt + swz_kv(np * 16 + (lane & 7) + ((lane >> 4) << 3), kk * 2 + ((lane >> 3) & 1)), b0, b1, b2, b3);
            mma_16816<E>(s[2 * np], qf[kk], b0, b1);
            mma_16816<E>(s[2 * np + 1], qf[kk], b2, b3);
          }
        }
        if (j0 + AT_KEYS > warp_first || row0 + 16 > rows) {   // the diagonal tiles (uniform over the warp)
#pragma unroll
          for (int nt = 0; nt < AT_KEYS / 8; ++nt) {
            const int j = j0 + nt * 8 + tq * 2;
            if (j >= lim_lo) s[nt][0] = -INFINITY;
            if (j + 1 >= lim_lo) s[nt][1] = -INFINITY;
            if (j >= lim_hi) s[nt][2] = -INFINITY;
            if (j + 1 >= lim_hi) s[nt][3] = -INFINITY;
          }
        }
        float mx_lo = -INFINITY, mx_hi = -INFINITY;
#pragma unroll
        for (int nt = 0; nt < AT_KEYS / 8; ++nt) {
          mx_lo = fmaxf(mx_lo, fmaxf(s[nt][0], s[nt][1]));
          mx_hi = fmaxf(mx_hi, fmaxf(s[nt][2], s[nt][3]));
        }
        mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 1));
        mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 2));
        mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 1));
        mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 2));
        const float mn_lo = fmaxf(m_lo, mx_lo * sl2), mn_hi = fmaxf(m_hi, mx_hi * sl2);
        const float ref_lo = (mn_lo == -INFINITY) ? 0.f : mn_lo, ref_hi = (mn_hi == -INFINITY) ? 0.f : mn_hi;
        const float al_lo = exp2f(m_lo - ref_lo), al_hi = exp2f(m_hi - ref_hi);
        m_lo = mn_lo; m_hi = mn_hi;
        float sum_lo = 0.f, sum_hi = 0.f;
#pragma unroll
        for (int nt = 0; nt < AT_KEYS / 8; ++nt) {
          s[nt][0] = exp2f(fmaf(s[nt][0], sl2, -ref_lo)); s[nt][1] = exp2f(fmaf(s[nt][1], sl2, -ref_lo));
          s[nt][2] = exp2f(fmaf(s[nt][2], sl2, -ref_hi)); s[nt][3] = exp2f(fmaf(s[nt][3], sl2, -ref_hi));
          sum_lo += s[nt][0] + s[nt][1];
          sum_hi += s[nt][2] + s[nt][3];
        }
        l_lo = l_lo * al_lo + sum_lo;
        l_hi = l_hi * al_hi + sum_hi;
#pragma unroll
        for (int i = 0; i < D / 8; ++i) { o[i][0] *= al_lo; o[i][1] *= al_lo; o[i][2] *= al_hi; o[i][3] *= al_hi; }
#pragma unroll
        for (int kk = 0; kk < AT_KEYS / 16; ++kk) {
          uint32_t pa[4];
          pa[0] = pack2<E>(s[2 * kk][0], s[2 * kk][1]);
          pa[1] = pack2<E>(s[2 * kk][2], s[2 * kk][3]);
          pa[2] = pack2<E>(s[2 * kk + 1][0], s[2 * kk + 1][1]);
          pa[3] = pack2<E>(s[2 * kk + 1][2], s[2 * kk + 1][3]);
#pragma unroll
          for (int dp = 0; dp < D / 16; ++dp) {
            uint32_t b0, b1, b2, b3;
            ldsm_x4_t(vt + swz_kv(kk * 16 + (lane & 7) + (((lane >> 3) & 1) << 3), dp * 2 + (lane >> 4)), b0, b1, b2, b3);
            mma_16816<E>(o[2 * dp], pa, b0, b1);
            mma_16816<E>(o[2 * dp + 1], pa, b2, b3);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty_bar(stage));
    }
    if (!ok && lane == 0 && p.status) atomicCAS(p.status, 0, ST_ATTENTION);
    l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1);
    l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
    l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1);
    l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int r = half ? r_hi : r_lo;
      if (r >= rows || !ok) continue;
      const float inv = 1.f / (half ? l_hi : l_lo);
      const size_t idx = ((size_t)(i0 + r) * p.hq + head) * D + tq * 2;
#pragma unroll
      for (int dt = 0; dt < D / 8; ++dt) {
        const float v0 = o[dt][2 * half] * inv, v1 = o[dt][2 * half + 1] * inv;
        uint32_t* dst = reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned short*>(p.out) + idx + dt * 8);
        if (p.fmt == XF_F16) {
          *dst = (uint32_t)f16_bits_sat(v0) | ((uint32_t)f16_bits_sat(v1) << 16);
        } else {
          const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
          *dst = *reinterpret_cast<const uint32_t*>(&h);
          if (p.fmt == XF_BF16X2) {
            const __nv_bfloat162 l = __floats2bfloat162_rn(v0 - __low2float(h), v1 - __high2float(h));
            *reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned short*>(p.out) + p.lo_off + idx + dt * 8) = *reinterpret_cast<const uint32_t*>(&l);
          }
        }
      }
    }
  }
  __syncthreads();     // the producer's copies have all been consumed (or drained) before any thread leaves
}

template <int D, typename E>
static cudaError_t pa_launch_t(const PaParams& p, cudaStream_t st) {
  using S = PaSmem<D>;
  static bool attr_set[MAX_DEVICES] = {};
  cudaError_t e = ensure_dynamic_smem(prefill_attn_kernel<D, E>, S::TOTAL, attr_set);
  if (e != cudaSuccess) return e;
  return launch_pdl(prefill_attn_kernel<D, E>, dim3(p.hq, ceil_div(p.n, S::ROWS)), dim3(S::THREADS), (size_t)S::TOTAL, st, p);
}

cudaError_t launch_prefill_attention(const AttnArgs& a, cudaStream_t st) {
  PaParams p;
  memset(&p, 0, sizeof(p));
  const int kind = a.kv_type == KV_F16 ? TM_F16 : TM_BF16;
  if (!make_tmap(&p.tm_k, a.kc, a.hkv * a.max_seq, a.d, AT_KEYS, kind) || !make_tmap(&p.tm_v, a.vc, a.hkv * a.max_seq, a.d, AT_KEYS, kind))
    return cudaErrorInvalidValue;
  p.q = a.q; p.out = a.out; p.lo_off = a.out_lo_off; p.fmt = a.out_fmt;
  p.n = a.n; p.L = a.cache_len; p.max_seq = a.max_seq; p.hq = a.hq; p.hkv = a.hkv; p.status = a.status;
  if (a.kv_type == KV_F16) return a.d == 128 ? pa_launch_t<128, __half>(p, st) : pa_launch_t<64, __half>(p, st);
  return a.d == 128 ? pa_launch_t<128, bf16>(p, st) : pa_launch_t<64, bf16>(p, st);
}

}  // namespace fdk
