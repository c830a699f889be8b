// The exact fp32 path: CUDA-core kernels of the decoder for fp32 weights (TF32 would miss its 1e-4 bound).
//
// Such models are small and their weights sit in L2: a forward is bound by the number of launches and by the round trips
// to memory inside each.  So a layer is five launches (projections finish what follows them: norm factor, bias, rotary and
// K / V rows, SwiGLU, residual), every load of a kernel is in flight at once, and the weights are on their way before the
// wait for the predecessor.  (One kernel per operator with split-K partial sums took 426 us for a step of the 2-layer,
// 256-wide shape with 8 rows; this takes 65 us, host round trip included.)
#include "kernels.h"

namespace fdk {

constexpr int FL_WARPS = 8;
constexpr int FL_KC = 1024;        // k values of the rows that are staged in shared memory at a time
constexpr int FL_STEP = 16 * FL_WARPS;
constexpr int FL_AHEAD = 6;        // k-steps whose weights are requested before the wait: 768 k

__device__ __forceinline__ float dot4(const float4& a, const float4& b, float c) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
}

// Four consecutive floats; `vec`: they are 16-byte aligned (callers' gains, queries and caches may lie at any float).
__device__ __forceinline__ float4 ldg_f4(const float* p, bool vec) {
  return vec ? __ldg(reinterpret_cast<const float4*>(p)) : make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}
__device__ __forceinline__ float4 ldcg_f4(const float* p, bool vec) {
  return vec ? __ldcg(reinterpret_cast<const float4*>(p)) : make_float4(__ldcg(p), __ldcg(p + 1), __ldcg(p + 2), __ldcg(p + 3));
}
static inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// What follows the sums a, b of features f0, f1 of row r (not LOGITS)
template <int MODE>
__device__ __forceinline__ void fl_finish(const F32Linear& p, int r, int mi, int f0, int f1, float a, float b) {
  if (MODE == FL_QKV) {
    const int half = p.d >> 1, j = f0 % p.d, head = f0 / p.d;
    const int pos0 = p.len_ptr ? *p.len_ptr : p.pos0;
    if (p.bias[mi]) { a += p.bias[mi][f0]; b += p.bias[mi][f1]; }
    if (mi < 2) {
      const float2 c = reinterpret_cast<const float2*>(p.cs)[(size_t)r * half + j];
      const float a0 = a, b0 = b;
      a = a0 * c.x - b0 * c.y;
      b = b0 * c.x + a0 * c.y;
    }
    float* dst = mi == 0 ? p.out + ((size_t)r * p.hq + head) * p.d + j
                         : (mi == 1 ? p.kc : p.vc) + ((size_t)head * p.max_seq + pos0 + r) * p.d + j;
    dst[0] = a;
    dst[half] = b;
  } else if (MODE == FL_SWIGLU) {
    if (f0 < p.n[0]) p.out[(size_t)r * p.n[0] + f0] = a / (1.f + expf(-a)) * b;
  } else {
    float* o = p.out + (size_t)r * p.n[0];
    if (f0 < p.n[0]) o[f0] += a;
    if (f1 < p.n[0]) o[f1] += b;
  }
}

// One CTA: RM rows x 8 pairs of output features.  The pair is what the epilogue combines: (j, j + d/2) of a head for the
// rotary embedding, (gate, up) for SwiGLU, else features f and f + 8.  GV: the gains are 16-byte aligned.  A warp takes every eighth 16-wide slice of k; lane =
// (feature 0..7, quarter of the slice).
template <int RM, int MODE, bool GV>
__global__ void __launch_bounds__(FL_WARPS * 32) linear_f32_kernel(const F32Linear p) {
  extern __shared__ float4 fl_smem[];
  float* xs = reinterpret_cast<float*>(fl_smem);                 // [RM][kc]
  __shared__ float red[FL_WARPS][RM][16];
  __shared__ float rstd[RM];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, fl = lane >> 2, kq = lane & 3;
  const int r0 = blockIdx.y * RM, K = p.k;
  const int kc = K < FL_KC ? K : FL_KC;
  pdl_trigger();
  // the two weight rows of this lane, and what the epilogue thread (row t / 8, pair t % 8) will need
  int mi = 0, f0, f1;
  auto pair_of = [&](int i) {
    if (MODE == FL_QKV) {
      const int half = p.d >> 1, tph = half / 8, head = blockIdx.x / tph;
      mi = head < p.hq ? 0 : (head < p.hq + p.hkv ? 1 : 2);
      const int hl = head - (mi == 0 ? 0 : (mi == 1 ? p.hq : p.hq + p.hkv));
      f0 = hl * p.d + (blockIdx.x % tph) * 8 + i;
      f1 = f0 + half;
    } else if (MODE == FL_SWIGLU) {
      f0 = f1 = blockIdx.x * 8 + i;
    } else {
      f0 = blockIdx.x * 16 + i;
      f1 = f0 + 8;
    }
  };
  pair_of(fl);
  const float* w0 = p.w[mi] + (size_t)min(f0, p.n[mi] - 1) * K;
  const float* w1 = (MODE == FL_SWIGLU ? p.w[1] : p.w[mi]) + (size_t)min(f1, p.n[mi] - 1) * K;
  float4 wa[FL_AHEAD], wb[FL_AHEAD];
#pragma unroll
  for (int s = 0; s < FL_AHEAD; ++s) {
    const int k = s * FL_STEP + warp * 16 + kq * 4;
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    wa[s] = k < K ? __ldg(reinterpret_cast<const float4*>(w0 + k)) : z;
    wb[s] = k < K ? __ldg(reinterpret_cast<const float4*>(w1 + k)) : z;
  }
  pdl_wait();
  float acc[RM][2], ssq[RM / FL_WARPS];
#pragma unroll
  for (int r = 0; r < RM; ++r) acc[r][0] = acc[r][1] = 0.f;
#pragma unroll
  for (int i = 0; i < RM / FL_WARPS; ++i) ssq[i] = 0.f;
  for (int c0 = 0; c0 < K; c0 += FL_KC) {
    const int cn = min(FL_KC, K - c0);
    if (c0) __syncthreads();
    // stage: warp w takes rows w, w + 8, ...
#pragma unroll
    for (int i = 0; i < RM / FL_WARPS; ++i) {
      const int rl = warp + i * FL_WARPS, r = r0 + rl;
      const float* src = p.x + (size_t)r * K + c0;
      float4 v[FL_KC / 128];
#pragma unroll
      for (int j = 0; j < FL_KC / 128; ++j) {
        const int k = lane * 4 + j * 128;
        v[j] = (r < p.m && k < cn) ? __ldcg(reinterpret_cast<const float4*>(src + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int j = 0; j < FL_KC / 128; ++j) {
        const int k = lane * 4 + j * 128;
        if (k >= cn) break;
        ssq[i] = dot4(v[j], v[j], ssq[i]);
        if (p.gain) {
          const float4 g = ldg_f4(p.gain + c0 + k, GV);
          v[j] = make_float4(v[j].x * g.x, v[j].y * g.y, v[j].z * g.z, v[j].w * g.w);
        }
        *reinterpret_cast<float4*>(xs + rl * kc + k) = v[j];
      }
    }
    __syncthreads();
    auto step = [&](int k, const float4& a, const float4& b) {
      const float* xp = xs + (k - c0);
#pragma unroll
      for (int r = 0; r < RM; ++r) {
        const float4 xv = *reinterpret_cast<const float4*>(xp + r * kc);
        acc[r][0] = dot4(a, xv, acc[r][0]);
        acc[r][1] = dot4(b, xv, acc[r][1]);
      }
    };
    int s = 0;
    if (c0 == 0) {
#pragma unroll
      for (s = 0; s < FL_AHEAD; ++s) {
        const int k = s * FL_STEP + warp * 16 + kq * 4;
        if (k < cn) step(k, wa[s], wb[s]);
      }
    }
#pragma unroll 2
    for (int k = c0 + s * FL_STEP + warp * 16 + kq * 4; k < c0 + cn; k += FL_STEP)
      step(k, __ldg(reinterpret_cast<const float4*>(w0 + k)), __ldg(reinterpret_cast<const float4*>(w1 + k)));
  }
  if (p.gain) {
#pragma unroll
    for (int i = 0; i < RM / FL_WARPS; ++i) {
      const float t = warp_sum(ssq[i]);
      if (lane == 0) rstd[warp + i * FL_WARPS] = rsqrtf(t * p.inv_h + p.eps);
    }
  }
#pragma unroll
  for (int r = 0; r < RM; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      float t = acc[r][c];
      t += __shfl_xor_sync(0xffffffffu, t, 1);
      t += __shfl_xor_sync(0xffffffffu, t, 2);
      if (kq == 0) red[warp][r][c * 8 + fl] = t;
    }
  __syncthreads();
  const int rl = threadIdx.x >> 3, i = threadIdx.x & 7, r = r0 + rl;
  if (rl >= RM) return;
  pair_of(i);
  float a = 0.f, b = 0.f;
#pragma unroll
  for (int w = 0; w < FL_WARPS; ++w) { a += red[w][rl][i]; b += red[w][rl][8 + i]; }
  if (p.gain) { a *= rstd[rl]; b *= rstd[rl]; }
  if (MODE == FL_LOGITS) {
    const bool in0 = f0 < p.n[0], in1 = f1 < p.n[0];
    if (p.out && r < p.m) {
      if (in0) p.out[(size_t)r * p.n[0] + f0] = a;
      if (in1) p.out[(size_t)r * p.n[0] + f1] = b;
    }
    if (!p.stats) return;
    // softmax statistics of the CTA's 16 vocabulary ids, the mask token excluded
    const float la = (in0 && f0 != p.mask_id) ? a : -INFINITY, lb = (in1 && f1 != p.mask_id) ? b : -INFINITY;
    float mx = fmaxf(fmaxf(la, lb), -INFINITY);       // (a NaN logit is no maximum; it does reach the sum)
    int ix = (lb > la || la != la) ? f1 : f0;         // (f0 < f1: a tie goes to the lower id)
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const float omx = __shfl_xor_sync(0xffffffffu, mx, o);
      const int oix = __shfl_xor_sync(0xffffffffu, ix, o);
      if (omx > mx || (omx == mx && oix < ix)) { mx = omx; ix = oix; }
    }
    float e = mx > -INFINITY ? __expf(la - mx) + __expf(lb - mx) : 0.f;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (i == 0 && r < p.m) p.stats[(size_t)blockIdx.x * p.m + r] = make_float4(mx, e, __int_as_float(ix), 0.f);
    return;
  }
  if (r >= p.m) return;
  fl_finish<MODE>(p, r, mi, f0, f1, a, b);
}

// The same for 32 rows x 16 pairs, two pairs per lane, where those CTAs still fill the SMs: with 32 rows the reads of a row's values from shared
// memory, one for every pair of a lane, bound the kernel above.  Step of 3 layers of the 3B shape in fp32, empty cache, one pair : two per lane:
// 32 rows 1453 : 1234 us, 33 rows 2338 : 1967, 64 rows 2500 : 2076; 1024 wide, 4 layers, 64 rows 839 : 747.  (A kernel of its own: as one
// source for both the kernels of 8 rows compiled to other register counts, and 1 row of the 3B shape went from 541 to 565 us.)
constexpr int FLW_ROWS = 32, FLW_PAIRS = 16;
template <int MODE, bool GV>
__global__ void __launch_bounds__(FL_WARPS * 32) linear_f32_wide_kernel(const F32Linear p) {
  extern __shared__ float4 fl_smem[];
  float* xs = reinterpret_cast<float*>(fl_smem);                 // [rows][kc]
  __shared__ float red[FL_WARPS][FLW_ROWS][2 * FLW_PAIRS];
  __shared__ float rstd[FLW_ROWS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, fl = lane >> 2, kq = lane & 3;
  const int r0 = blockIdx.y * FLW_ROWS, K = p.k;
  const int kc = K < FL_KC ? K : FL_KC;
  pdl_trigger();
  int mi = 0, f0, f1;
  auto pair_of = [&](int i) {
    if (MODE == FL_QKV) {
      const int half = p.d >> 1, tph = half / FLW_PAIRS, head = blockIdx.x / tph;
      mi = head < p.hq ? 0 : (head < p.hq + p.hkv ? 1 : 2);
      const int hl = head - (mi == 0 ? 0 : (mi == 1 ? p.hq : p.hq + p.hkv));
      f0 = hl * p.d + (blockIdx.x % tph) * FLW_PAIRS + i;
      f1 = f0 + half;
    } else if (MODE == FL_SWIGLU) {
      f0 = f1 = blockIdx.x * FLW_PAIRS + i;
    } else {
      f0 = blockIdx.x * (2 * FLW_PAIRS) + i;
      f1 = f0 + FLW_PAIRS;
    }
  };
  const float* wp[4];              // first and second feature of pairs fl and fl + 8
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    pair_of(fl + 8 * q);
    wp[2 * q] = p.w[mi] + (size_t)min(f0, p.n[mi] - 1) * K;
    wp[2 * q + 1] = (MODE == FL_SWIGLU ? p.w[1] : p.w[mi]) + (size_t)min(f1, p.n[mi] - 1) * K;
  }
  pdl_wait();
  float acc[FLW_ROWS][4], ssq[FLW_ROWS / FL_WARPS];
#pragma unroll
  for (int r = 0; r < FLW_ROWS; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0.f;
#pragma unroll
  for (int i = 0; i < FLW_ROWS / FL_WARPS; ++i) ssq[i] = 0.f;
  for (int c0 = 0; c0 < K; c0 += FL_KC) {
    const int cn = min(FL_KC, K - c0);
    if (c0) __syncthreads();
#pragma unroll
    for (int i = 0; i < FLW_ROWS / FL_WARPS; ++i) {
      const int rl = warp + i * FL_WARPS, r = r0 + rl;
      const float* src = p.x + (size_t)r * K + c0;
      float4 v[FL_KC / 128];
#pragma unroll
      for (int j = 0; j < FL_KC / 128; ++j) {
        const int k = lane * 4 + j * 128;
        v[j] = (r < p.m && k < cn) ? __ldcg(reinterpret_cast<const float4*>(src + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int j = 0; j < FL_KC / 128; ++j) {
        const int k = lane * 4 + j * 128;
        if (k >= cn) break;
        ssq[i] = dot4(v[j], v[j], ssq[i]);
        if (p.gain) {
          const float4 g = ldg_f4(p.gain + c0 + k, GV);
          v[j] = make_float4(v[j].x * g.x, v[j].y * g.y, v[j].z * g.z, v[j].w * g.w);
        }
        *reinterpret_cast<float4*>(xs + rl * kc + k) = v[j];
      }
    }
    __syncthreads();
#pragma unroll 2
    for (int k = c0 + warp * 16 + kq * 4; k < c0 + cn; k += FL_STEP) {
      float4 w[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) w[c] = __ldg(reinterpret_cast<const float4*>(wp[c] + k));
      const float* xp = xs + (k - c0);
#pragma unroll
      for (int r = 0; r < FLW_ROWS; ++r) {
        const float4 xv = *reinterpret_cast<const float4*>(xp + r * kc);
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = dot4(w[c], xv, acc[r][c]);
      }
    }
  }
  if (p.gain) {
#pragma unroll
    for (int i = 0; i < FLW_ROWS / FL_WARPS; ++i) {
      const float t = warp_sum(ssq[i]);
      if (lane == 0) rstd[warp + i * FL_WARPS] = rsqrtf(t * p.inv_h + p.eps);
    }
  }
#pragma unroll
  for (int r = 0; r < FLW_ROWS; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float t = acc[r][c];
      t += __shfl_xor_sync(0xffffffffu, t, 1);
      t += __shfl_xor_sync(0xffffffffu, t, 2);
      if (kq == 0) red[warp][r][(c & 1) * FLW_PAIRS + (c >> 1) * 8 + fl] = t;
    }
  __syncthreads();
  // thread: row t / 8, pairs t % 8 and 8 further on
  const int rl = threadIdx.x >> 3, i = threadIdx.x & 7, r = r0 + rl;
  [[maybe_unused]] float lv[4], mx = -INFINITY;       // LOGITS: this thread's logits that count, their maximum (a NaN is none) and its id
  [[maybe_unused]] int ix = 0x7fffffff;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    pair_of(i + 8 * q);
    float v[2] = {0.f, 0.f};
#pragma unroll
    for (int w = 0; w < FL_WARPS; ++w)
#pragma unroll
      for (int c = 0; c < 2; ++c) v[c] += red[w][rl][c * FLW_PAIRS + 8 * q + i];
    if (p.gain) { v[0] *= rstd[rl]; v[1] *= rstd[rl]; }
    if constexpr (MODE != FL_LOGITS) {
      if (r < p.m) fl_finish<MODE>(p, r, mi, f0, f1, v[0], v[1]);
    } else {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int f = c ? f1 : f0;
        const bool in = f < p.n[0];
        if (p.out && in && r < p.m) p.out[(size_t)r * p.n[0] + f] = v[c];
        const float l = (in && f != p.mask_id) ? v[c] : -INFINITY;
        lv[2 * q + c] = l;
        if (l > mx || (l == mx && f < ix)) { mx = l; ix = f; }      // (a tie goes to the lower id)
      }
    }
  }
  if constexpr (MODE == FL_LOGITS) {
    if (!p.stats) return;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const float omx = __shfl_xor_sync(0xffffffffu, mx, o);
      const int oix = __shfl_xor_sync(0xffffffffu, ix, o);
      if (omx > mx || (omx == mx && oix < ix)) { mx = omx; ix = oix; }
    }
    float e = 0.f;
    if (mx > -INFINITY) {
#pragma unroll
      for (int c = 0; c < 4; ++c) e += __expf(lv[c] - mx);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (i == 0 && r < p.m) p.stats[(size_t)blockIdx.x * p.m + r] = make_float4(mx, e, __int_as_float(ix), 0.f);
  }
}

template <int RM>
static cudaError_t fl_launch(void (*kern)(F32Linear), bool* attr_set, const F32Linear& p, int tiles, cudaStream_t st) {
  cudaError_t e = ensure_dynamic_smem(kern, RM * FL_KC * 4, attr_set);
  if (e != cudaSuccess) return e;
  const size_t smem = (size_t)RM * (p.k < FL_KC ? p.k : FL_KC) * 4;
  return launch_pdl(kern, dim3(tiles, ceil_div(p.m, RM)), dim3(FL_WARPS * 32), smem, st, p);
}
template <int RM, int MODE>
static cudaError_t fl_launch_t(const F32Linear& p, int tiles, cudaStream_t st) {
  static bool attr_set[2][MAX_DEVICES] = {};
  return aligned16(p.gain) ? fl_launch<RM>(linear_f32_kernel<RM, MODE, true>, attr_set[0], p, tiles, st)
                           : fl_launch<RM>(linear_f32_kernel<RM, MODE, false>, attr_set[1], p, tiles, st);
}
template <int MODE>
static cudaError_t fl_launch_wide(const F32Linear& p, int tiles, cudaStream_t st) {
  static bool attr_set[2][MAX_DEVICES] = {};
  return aligned16(p.gain) ? fl_launch<FLW_ROWS>(linear_f32_wide_kernel<MODE, true>, attr_set[0], p, tiles, st)
                           : fl_launch<FLW_ROWS>(linear_f32_wide_kernel<MODE, false>, attr_set[1], p, tiles, st);
}
// whether m rows of `features` output features take the wide kernel
static bool fl_wide(int m, int features) {
  return m > 16 && ceil_div(features, 2 * FLW_PAIRS) * ceil_div(m, FLW_ROWS) >= sm_count();
}
// rows per CTA: all of them up to 32, so that a weight is read once (64 rows: twice)
template <int MODE>
static cudaError_t fl_launch_m(const F32Linear& p, int features, cudaStream_t st) {
  if (fl_wide(p.m, features)) return fl_launch_wide<MODE>(p, ceil_div(features, 2 * FLW_PAIRS), st);
  const int tiles = ceil_div(features, 16);
  if (p.m <= 8) return fl_launch_t<8, MODE>(p, tiles, st);
  if (p.m <= 16) return fl_launch_t<16, MODE>(p, tiles, st);
  return fl_launch_t<32, MODE>(p, tiles, st);
}
int f32_logit_tiles(int vocab, int m) { return ceil_div(vocab, fl_wide(m, vocab) ? 2 * FLW_PAIRS : 16); }
cudaError_t launch_linear_f32(const F32Linear& p, cudaStream_t st) {
  switch (p.mode) {
    case FL_QKV: return fl_launch_m<FL_QKV>(p, (p.hq + 2 * p.hkv) * p.d, st);
    case FL_SWIGLU: return fl_launch_m<FL_SWIGLU>(p, 2 * p.n[0], st);
    case FL_RESID: return fl_launch_m<FL_RESID>(p, p.n[0], st);
    default: return fl_launch_m<FL_LOGITS>(p, p.n[0], st);
  }
}

// ================================================================================================
// attention: one CTA per (query head, row), keys in chunks of FA_KEYS with an online softmax across chunks
// ================================================================================================
constexpr int FA_THREADS = 256, FA_KEYS = 2048, FA_U = 8;      // FA_U: loads in flight per thread

// VEC: q and the caches are 16-byte aligned
template <int D, bool VEC>
__global__ void __launch_bounds__(FA_THREADS) attn_f32_kernel(const float* __restrict__ q, const float* __restrict__ kc,
                                                              const float* __restrict__ vc, float* __restrict__ out, int n, int L,
                                                              const int* __restrict__ len_ptr, int max_seq, int hq, int hkv, int causal,
                                                              const unsigned long long* __restrict__ row_mask) {
  constexpr int LPK = D / 4, KPW = 32 / LPK, PARTS = FA_THREADS / LPK, NW = FA_THREADS / 32;
  __shared__ __align__(16) float sc[FA_KEYS];
  __shared__ __align__(16) float ov[PARTS][D];
  __shared__ float red[32];
  pdl_trigger();
  const int head = blockIdx.x, r = blockIdx.y, hk = head / (hq / hkv);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sub = lane / LPK, li = lane % LPK, part = threadIdx.x / LPK, col = threadIdx.x % LPK;
  if (len_ptr) L = *len_ptr;
  const int T = causal ? L + r + 1 : L + n;
  const float* kb = kc + (size_t)hk * max_seq * D;
  const float* vb = vc + (size_t)hk * max_seq * D;
  pdl_wait();
  const float scale = rsqrtf((float)D);
  float4 qv = ldcg_f4(q + ((size_t)r * hq + head) * D + li * 4, VEC);
  qv = make_float4(qv.x * scale, qv.y * scale, qv.z * scale, qv.w * scale);
  const unsigned long long mask = row_mask ? row_mask[r] : ~0ull;
  float m_run = -INFINITY, sum = 0.f;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int c0 = 0; c0 < T; c0 += FA_KEYS) {
    const int cn = min(FA_KEYS, T - c0);
    if (c0) __syncthreads();
    for (int b = warp * KPW * FA_U; b < cn; b += NW * KPW * FA_U) {
      float4 kv[FA_U];
#pragma unroll
      for (int u = 0; u < FA_U; ++u) kv[u] = ldcg_f4(kb + (size_t)(c0 + min(b + u * KPW + sub, cn - 1)) * D + li * 4, VEC);
#pragma unroll
      for (int u = 0; u < FA_U; ++u) {
        float s = dot4(qv, kv[u], 0.f);
#pragma unroll
        for (int o = LPK / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const int j = b + u * KPW + sub;
        // bit r' of the mask: this row reads row r' of the forward (the cache is always read)
        if (c0 + j >= L && !((mask >> (c0 + j - L)) & 1ull)) s = -INFINITY;
        if (li == 0 && j < cn) sc[j] = s;
      }
    }
    __syncthreads();
    float mx = -INFINITY;
    for (int j = threadIdx.x; j < cn; j += FA_THREADS) mx = fmaxf(mx, sc[j]);
    mx = fmaxf(m_run, block_max(mx, red));
    const float ref = mx == -INFINITY ? 0.f : mx, keep = expf(m_run - ref);
    m_run = mx;
    float cs = 0.f;
    for (int j = threadIdx.x; j < cn; j += FA_THREADS) {
      const float e = expf(sc[j] - ref);
      sc[j] = e;
      cs += e;
    }
    sum = sum * keep + block_sum(cs, red);
    __syncthreads();
    acc = make_float4(acc.x * keep, acc.y * keep, acc.z * keep, acc.w * keep);
    for (int j0 = part; j0 < cn; j0 += PARTS * FA_U) {
      float4 vv[FA_U];
#pragma unroll
      for (int u = 0; u < FA_U; ++u) vv[u] = ldcg_f4(vb + (size_t)(c0 + min(j0 + u * PARTS, cn - 1)) * D + col * 4, VEC);
#pragma unroll
      for (int u = 0; u < FA_U; ++u) {
        const int j = j0 + u * PARTS;
        const float w = j < cn ? sc[j] : 0.f;
        acc = make_float4(fmaf(w, vv[u].x, acc.x), fmaf(w, vv[u].y, acc.y), fmaf(w, vv[u].z, acc.z), fmaf(w, vv[u].w, acc.w));
      }
    }
  }
  *reinterpret_cast<float4*>(&ov[part][col * 4]) = acc;
  __syncthreads();
  if (threadIdx.x < D) {
    float o = 0.f;
#pragma unroll
    for (int i = 0; i < PARTS; ++i) o += ov[i][threadIdx.x];
    out[((size_t)r * hq + head) * D + threadIdx.x] = o / sum;
  }
}

int launch_attention_f32(const AttnArgs& a, cudaStream_t st, cudaError_t* err) {
  const bool vec = aligned16(a.q) && aligned16(a.kc) && aligned16(a.vc);
  auto kern = a.d == 128 ? (vec ? attn_f32_kernel<128, true> : attn_f32_kernel<128, false>) : (vec ? attn_f32_kernel<64, true> : attn_f32_kernel<64, false>);
  *err = launch_pdl(kern, dim3(a.hq, a.n), dim3(FA_THREADS), 0, st, (const float*)a.q, (const float*)a.kc, (const float*)a.vc, (float*)a.out,
                    a.n, a.cache_len, a.len_ptr, a.max_seq, a.hq, a.hkv, a.causal, a.row_mask);
  return *err == cudaSuccess ? 1 : -1;
}

}  // namespace fdk
