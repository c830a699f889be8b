// The small kernels of every configuration (embedding gather, rotary table, the glue of the tensor-core path, confidence
// statistics, unmask selection, block state) and the stand-alone CUDA-core projection.
#include "common.cuh"
#include "kernels.h"

namespace fdk {

// ================================================================================================
// small-M linear, CUDA-core version.  Register-tiled: CTA tile BM x 64 outputs, BK = 32 deep.
// Used for fp32 weights (TF32 tensor cores would miss the 1e-4 parity bound of that path) and for
// shapes the tensor-core kernel does not take.
// ================================================================================================
template <typename T> struct Vec8;
template <> struct Vec8<float> {
  static __device__ __forceinline__ void load(const float* p, float* o) {
    float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w; o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
  }
};
template <> struct Vec8<bf16> {
  static __device__ __forceinline__ void load(const bf16* p, float* o) {
    uint4 v = *reinterpret_cast<const uint4*>(p);
    const unsigned u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      o[2 * i] = __uint_as_float(u[i] << 16);
      o[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
    }
  }
};
template <> struct Vec8<fp8e4m3> {
  static __device__ __forceinline__ void load(const fp8e4m3* p, float* o) {
    uint2 v = *reinterpret_cast<const uint2*>(p);
    const unsigned u[2] = {v.x, v.y};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      fp8e4m3 e;
      e.b = (uint8_t)((u[i >> 2] >> (8 * (i & 3))) & 0xffu);
      o[i] = to_f32(e);
    }
  }
};

constexpr int SBN = 64, SBK = 32;

template <typename WT, typename XT, int BM>
__global__ void __launch_bounds__((BM / 4) * 16)
linear_simt_kernel(const XT* __restrict__ x, const WT* __restrict__ w, float* __restrict__ part,
                   int m, int N, int K, int k_per_split) {
  constexpr int NT = (BM / 4) * 16;
  __shared__ __align__(16) float xs[SBK][BM + 4];
  __shared__ __align__(16) float ws[SBK][SBN + 4];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int n0 = blockIdx.x * SBN;
  const int kb = blockIdx.y * k_per_split;
  const int ke = min(K, kb + k_per_split);
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

  for (int k0 = kb; k0 < ke; k0 += SBK) {
    // W tile: 64 rows x 32 k as 256 vectors of 8; vector v -> row v % 64, k-quarter v / 64
    for (int v = tid; v < SBN * (SBK / 8); v += NT) {
      int r = v % SBN, kq = v / SBN;
      int n = n0 + r, k = k0 + kq * 8;
      float f[8];
      if (n < N && k < ke) Vec8<WT>::load(w + (size_t)n * K + k, f);
      else {
#pragma unroll
        for (int i = 0; i < 8; ++i) f[i] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) ws[kq * 8 + i][r] = f[i];
    }
    for (int v = tid; v < BM * (SBK / 8); v += NT) {
      int r = v % BM, kq = v / BM;
      int k = k0 + kq * 8;
      float f[8];
      if (r < m && k < ke) Vec8<XT>::load(x + (size_t)r * K + k, f);
      else {
#pragma unroll
        for (int i = 0; i < 8; ++i) f[i] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) xs[kq * 8 + i][r] = f[i];
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < SBK; ++kk) {
      float4 xv = *reinterpret_cast<const float4*>(&xs[kk][ty * 4]);
      float4 wv = *reinterpret_cast<const float4*>(&ws[kk][tx * 4]);
      const float xa[4] = {xv.x, xv.y, xv.z, xv.w}, wa[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xa[i], wa[j], acc[i][j]);
    }
    __syncthreads();
  }
  float* dst = part + (size_t)blockIdx.y * m * N;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int r = ty * 4 + i;
    if (r >= m) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int n = n0 + tx * 4 + j;
      if (n < N) dst[(size_t)r * N + n] = acc[i][j];
    }
  }
}

// y[r, n] = (sum_s part[s][r][n]) * scale[n] + bias[n]; fixed summation order.
__global__ void splitk_epilogue_kernel(const float* __restrict__ part, int S, int m, int N,
                                       const float* __restrict__ scale, const float* __restrict__ bias,
                                       float* __restrict__ y, const float* __restrict__ x_scale) {
  pdl_trigger();
  pdl_wait();
  size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  size_t total = (size_t)m * N;
  if (idx >= total) return;
  int r = (int)(idx / N), n = (int)(idx % N);
  float s = 0.f;
  for (int i = 0; i < S; ++i) s += part[(size_t)i * total + idx];
  if (scale) s *= scale[n];
  if (x_scale) s *= x_scale[r];   // sums of e4m3 code products
  if (bias) s += bias[n];
  y[idx] = s;
}

void launch_splitk_epilogue(const float* part, int S, int m, int n, const float* scale, const float* bias, float* y,
                            cudaStream_t st, const float* x_scale) {
  size_t total = (size_t)m * n;
  splitk_epilogue_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(part, S, m, n, scale, bias, y, x_scale);
}

static void simt_plan(int m, int n, int k, int* bm, int* splits, int* kps) {
  *bm = m <= 16 ? 16 : (m <= 32 ? 32 : 64);
  int tiles = ceil_div(n, SBN);
  int kblocks = ceil_div(k, SBK);
  int want = ceil_div(2 * 148, tiles);                 // at least ~2 CTAs per SM when K allows
  int s = want < 1 ? 1 : want;
  int max_s = kblocks / 8 > 0 ? kblocks / 8 : 1;       // >= 256 deep per split
  if (s > max_s) s = max_s;
  if (s > 16) s = 16;
  int per = ceil_div(kblocks, s) * SBK;
  *kps = per;
  *splits = ceil_div(k, per);
}

size_t simt_workspace_bytes(int m, int n, int k) {
  int bm, s, kps;
  simt_plan(m, n, k, &bm, &s, &kps);
  return (size_t)s * m * n * sizeof(float);
}

template <typename WT, typename XT>
static void simt_dispatch(const LinearArgs& a, int bm, dim3 grid, float* part, int kps, cudaStream_t st) {
  const XT* x = (const XT*)a.x;
  const WT* w = (const WT*)a.w;
  if (bm == 16) linear_simt_kernel<WT, XT, 16><<<grid, 64, 0, st>>>(x, w, part, a.m, a.n, a.k, kps);
  else if (bm == 32) linear_simt_kernel<WT, XT, 32><<<grid, 128, 0, st>>>(x, w, part, a.m, a.n, a.k, kps);
  else linear_simt_kernel<WT, XT, 64><<<grid, 256, 0, st>>>(x, w, part, a.m, a.n, a.k, kps);
}

int launch_linear_simt(const LinearArgs& a, cudaStream_t st, cudaError_t* err) {
  int bm, s, kps;
  simt_plan(a.m, a.n, a.k, &bm, &s, &kps);
  size_t need = (size_t)s * a.m * a.n * sizeof(float);
  if (need > a.workspace_bytes || a.workspace == nullptr) { *err = cudaErrorInvalidValue; return -1; }
  float* part = (float*)a.workspace;
  dim3 grid(ceil_div(a.n, SBN), s);
  if (a.dtype == DT_F32) simt_dispatch<float, float>(a, bm, grid, part, kps, st);
  else if (a.dtype == DT_BF16) simt_dispatch<bf16, bf16>(a, bm, grid, part, kps, st);
  else simt_dispatch<fp8e4m3, bf16>(a, bm, grid, part, kps, st);
  size_t total = (size_t)a.m * a.n;
  splitk_epilogue_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(part, s, a.m, a.n, a.scale, a.bias, a.y,
                                                                         nullptr);
  *err = cudaGetLastError();
  return *err == cudaSuccess ? 2 : -1;
}

// ================================================================================================
// embedding gather / row conversion
// ================================================================================================
// A token id outside [0, vocab) is not dereferenced: row 0 is read instead and ST_BAD_TOKEN is left in the status word.
__device__ __forceinline__ int checked_token(const int32_t* tokens, int r, int vocab, int* status) {
  const int t = tokens[r];
  if (t >= 0 && t < vocab) return t;
  if (threadIdx.x == 0 && status) atomicCAS(status, 0, ST_BAD_TOKEN);
  return 0;
}
// fp32 rows into the residual stream: those of `tokens`, or (null) the first n of the table
__global__ void embed_f32_kernel(const float* __restrict__ table, const int32_t* __restrict__ tokens,
                                 float* __restrict__ h, int hidden, int vocab, int* status) {
  int r = blockIdx.x;
  const float* src = table + (size_t)(tokens ? checked_token(tokens, r, vocab, status) : r) * hidden;
  for (int c = threadIdx.x; c < hidden; c += blockDim.x) h[(size_t)r * hidden + c] = src[c];
}
void launch_embed_f32(const void* table, const int32_t* tokens, float* h, int n, int hidden, int vocab, int* status, cudaStream_t st) {
  embed_f32_kernel<<<n, 256, 0, st>>>((const float*)table, tokens, h, hidden, vocab, status);
}
// cs[r][j] = (cos, sin) of position(r) * theta^(-j / half), as rope_table_kernel below
__device__ __forceinline__ float2 rope_entry(int pos, int j, int half, double theta) {
  const double inv = pow(theta, -(double)j / (double)half);
  double s, c;
  sincos((double)pos * inv, &s, &c);
  return make_float2((float)c, (float)s);
}
// The embedding gather and the rotary table of one fp32 row block in one launch: both are a microsecond of latency, so the launch is
// what they cost.  With the selection captured too, a step from the host is one graph launch (8 rows of the tiny shape: 62 -> 55 us a step,
// commit of a block 54 -> 49).
__global__ void embed_rope_f32_kernel(const float* __restrict__ table, const int32_t* __restrict__ tokens, float* __restrict__ h, int hidden,
                                      int vocab, int* status, float2* __restrict__ cs, int pos0, int half, double theta,
                                      const int* __restrict__ len_ptr, const int* __restrict__ pos_off) {
  pdl_trigger();
  pdl_wait();
  const int r = blockIdx.x;
  const float* src = table + (size_t)checked_token(tokens, r, vocab, status) * hidden;
  for (int c = threadIdx.x; c < hidden; c += blockDim.x) h[(size_t)r * hidden + c] = src[c];
  if (len_ptr) pos0 = *len_ptr;
  for (int j = threadIdx.x; j < half; j += blockDim.x) cs[r * half + j] = rope_entry(pos0 + (pos_off ? pos_off[r] : r), j, half, theta);
}
void launch_embed_rope_f32(const void* table, const int32_t* tokens, float* h, int n, int hidden, int vocab, int* status, float* cs,
                           int pos0, int head_dim, float theta, const int* len_ptr, const int* pos_off, cudaStream_t st) {
  launch_pdl(embed_rope_f32_kernel, dim3(n), dim3(128), 0, st, (const float*)table, tokens, h, hidden, vocab, status, (float2*)cs, pos0,
             head_dim / 2, (double)theta, len_ptr, pos_off);
}

// ================================================================================================
// rotary table: cs[r][j] = (cos, sin)(pos * theta^(-2j/d)), angles formed in fp64
// ================================================================================================
__global__ void set_len_kernel(int* len_ptr, int value) {
  pdl_trigger();
  pdl_wait();
  *len_ptr = value;
}
void launch_set_len(int* len_ptr, int value, cudaStream_t st) { set_len_kernel<<<1, 1, 0, st>>>(len_ptr, value); }

// cs[r][j] = (cos, sin) of position(r) * theta^(-j / half); position(r) = pos0 + r, or pos0 + pos_off[r] when the rows
// carry their own position ids (Appendix B, Alg. 2: group i of the quadratic input covers positions s+i .. s+i+B)
__global__ void rope_table_kernel(float2* __restrict__ cs, int n, int pos0, int half, double theta, const int* __restrict__ len_ptr,
                                  const int* __restrict__ pos_off, KStamp* stamp) {
  if (threadIdx.x == 0) stamp_start(stamp);
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) { stamp_released(stamp); stamp_end(stamp); }
  if (len_ptr) pos0 = *len_ptr;
  int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n * half) return;
  int r = idx / half, j = idx % half;
  cs[idx] = rope_entry(pos0 + (pos_off ? pos_off[r] : r), j, half, theta);
}
void launch_rope_table(float* cs, int n, int pos0, int head_dim, float theta, cudaStream_t st, const int* len_ptr, KStamp* stamp,
                       const int* pos_off) {
  int half = head_dim / 2, total = n * half;
  launch_pdl(rope_table_kernel, dim3((total + 127) / 128), dim3(128), 0, st, (float2*)cs, n, pos0, half, (double)theta, len_ptr, pos_off,
             stamp);
}

// ================================================================================================
// Glue of the tensor-core path.  RMSNorm is folded into its consumer GEMM: producers leave xg = h * gain as a GEMM
// input (XF_* storage: bf16 hi + lo planes, or f16) and per-128-column partial sums of h^2 (ssq[row][nt]); the
// consumer's epilogue multiplies by rsqrt(sum(ssq) / hidden + eps).  All sums run in a fixed order => deterministic.
// ================================================================================================
// W8A8 (Sec. 3.4 "System integration"): a projection input row is quantised to e4m3 with the scale max|row| / 448, the
// maximum taken over the values as stored (f16).  Producers leave partial maxima; consumers of code-product sums
// multiply by the scale.
__device__ __forceinline__ float abs_as_f16(float v) { return fabsf(__half2float(__ushort_as_half(f16_bits_sat(v)))); }
__device__ __forceinline__ float scale_of_amax(float amax) { return amax > 0.f ? __fdiv_rn(amax, 448.f) : 1.f; }

__global__ void embed_prep_kernel(const bf16* __restrict__ table, const int32_t* __restrict__ tokens,
                                  const bf16* __restrict__ rows, float* __restrict__ h, void* __restrict__ xg,
                                  size_t lo_off, int fmt, const float* __restrict__ g, float* __restrict__ ssq, int nt,
                                  int hidden, int vocab, int* status, float* __restrict__ amax, KStamp* stamp) {
  if (threadIdx.x == 0) stamp_start(stamp);
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) stamp_released(stamp);
  __shared__ float red[32];
  const int r = blockIdx.x;
  const bf16* src = tokens ? table + (size_t)checked_token(tokens, r, vocab, status) * hidden : rows + (size_t)r * hidden;
  float ss = 0.f, am = 0.f;
  for (int c = threadIdx.x; c < hidden; c += blockDim.x) {
    const float v = __bfloat162float(src[c]);
    h[(size_t)r * hidden + c] = v;
    store_act(xg, lo_off, (size_t)r * hidden + c, v * g[c], fmt);
    ss = fmaf(v, v, ss);
    am = fmaxf(am, abs_as_f16(v * g[c]));
  }
  ss = block_sum(ss, red);
  for (int t = threadIdx.x; t < nt; t += blockDim.x) ssq[(size_t)r * nt + t] = (t == 0) ? ss : 0.f;
  if (amax) {      // same layout as ssq: the whole row's maximum in slot 0
    __syncthreads();
    am = block_max(am, red);
    for (int t = threadIdx.x; t < nt; t += blockDim.x) amax[(size_t)r * nt + t] = (t == 0) ? am : 0.f;
  }
  if (threadIdx.x == 0) stamp_end(stamp);
}
void launch_embed_prep(const void* table, const int32_t* tokens, const void* rows, float* h, void* xg, size_t lo_off, int fmt,
                       const float* g, float* ssq, int nt, int n, int hidden, int vocab, int* status, cudaStream_t st, KStamp* stamp,
                       float* amax) {
  embed_prep_kernel<<<n, 256, 0, st>>>((const bf16*)table, tokens, (const bf16*)rows, h, xg, lo_off, fmt, g, ssq, nt, hidden, vocab,
                                       status, amax, stamp);
}

// bf16 rows -> the planes of XF_E5M2X3, n bytes apart, for the operator-level entry points whose callers hand bf16
// activations to an fp8-weight projection
__global__ void bf16_to_e5m2x3_kernel(const bf16* __restrict__ in, uint8_t* __restrict__ out, size_t n) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) store_act(out, n, i, __bfloat162float(in[i]), XF_E5M2X3);
}
void launch_bf16_to_e5m2x3(const void* in, void* out, size_t n, cudaStream_t st) {
  bf16_to_e5m2x3_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const bf16*)in, (uint8_t*)out, n);
}
// Eight f16 values -> e4m3 codes of x / scale: float32 quotient, round to nearest even, saturating.  The quotient is formed
// without the division routine: with y = RN(1 / scale), q0 = RN(x y) and the exact remainder r = x - q0 scale (one FMA),
// RN(q0 + r y) is the correctly rounded x / scale (Markstein's correction step; no operand here is zero, infinite or
// subnormal except x = 0, which gives 0 either way).
__device__ __forceinline__ uint2 e4m3_codes8(uint4 x, float sc, float rinv) {
  const uint32_t in[4] = {x.x, x.y, x.z, x.w};
  unsigned short out[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&in[i]));
    const float q0 = a.x * rinv, q1 = a.y * rinv;
    const float x0 = fmaf(fmaf(-q0, sc, a.x), rinv, q0), x1 = fmaf(fmaf(-q1, sc, a.y), rinv, q1);
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(out[i]) : "f"(x1), "f"(x0));   // first source -> upper byte
  }
  return make_uint2((uint32_t)out[0] | ((uint32_t)out[1] << 16), (uint32_t)out[2] | ((uint32_t)out[3] << 16));
}
// grid (ceil(k / 1024), rows), 128 threads, eight values each: two dependent L2 round trips, of which the maxima and the values share
// the first, so the launch and those are what it costs (about 2 us) and more values a thread would only lengthen it.  Against quantising in the
// projections' own warps: 8 layers of the 7B shape and the LM head 843 -> 731 us a step at 32 rows, 717 -> 657 at 8.
__global__ void __launch_bounds__(128) quantize_rows_kernel(const unsigned short* __restrict__ x, int k, const float* __restrict__ amax,
                                                            int n_amax, uint8_t* __restrict__ codes, float* __restrict__ scale) {
  pdl_trigger();
  pdl_wait();
  const int r = blockIdx.y, c = (blockIdx.x * 128 + threadIdx.x) * 8, lane = threadIdx.x & 31;
  uint4 v = make_uint4(0, 0, 0, 0);
  if (c < k) v = __ldcg(reinterpret_cast<const uint4*>(x + (size_t)r * k + c));
  float am = 0.f;
  for (int i = lane; i < n_amax; i += 32) am = fmaxf(am, __ldcg(amax + (size_t)r * n_amax + i));
  const float sc = scale_of_amax(warp_max(am));
  if (c < k) *reinterpret_cast<uint2*>(codes + (size_t)r * k + c) = e4m3_codes8(v, sc, __frcp_rn(sc));
  if (blockIdx.x == 0 && threadIdx.x == 0) scale[r] = sc;
}
void launch_quantize_rows(const void* x, int m, int k, const float* amax, int n_amax, void* codes, float* scale, cudaStream_t st) {
  launch_pdl(quantize_rows_kernel, dim3((k + 1023) / 1024, m), dim3(128), 0, st, (const unsigned short*)x, k, amax, n_amax,
             (uint8_t*)codes, scale);
}
__global__ void __launch_bounds__(256) quantize_bf16_rows_kernel(const bf16* __restrict__ in, int k, uint8_t* __restrict__ codes,
                                                                 float* __restrict__ scale) {
  __shared__ float red[32];
  const size_t base = (size_t)blockIdx.x * k;
  float am = 0.f;
  for (int c = threadIdx.x; c < k; c += blockDim.x) am = fmaxf(am, abs_as_f16(__bfloat162float(in[base + c])));
  const float sc = scale_of_amax(block_max(am, red)), rinv = __frcp_rn(sc);
  for (int c = threadIdx.x * 8; c < k; c += blockDim.x * 8) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      w[i] = (uint32_t)f16_bits_sat(__bfloat162float(in[base + c + 2 * i])) | ((uint32_t)f16_bits_sat(__bfloat162float(in[base + c + 2 * i + 1])) << 16);
    *reinterpret_cast<uint2*>(codes + base + c) = e4m3_codes8(make_uint4(w[0], w[1], w[2], w[3]), sc, rinv);
  }
  if (threadIdx.x == 0) scale[blockIdx.x] = sc;
}
void launch_quantize_bf16_rows(const void* in, int m, int k, void* codes, float* scale, cudaStream_t st) {
  quantize_bf16_rows_kernel<<<m, 256, 0, st>>>((const bf16*)in, k, (uint8_t*)codes, scale);
}

// Sums of S split-K partials, V consecutive columns a lane.  These kernels are a handful of dependent L2 round trips long, so every
// load that can be issued at once is: NP partials in flight, added in index order (deterministic).
template <int V> struct Cols { float v[V]; };
template <int V>
__device__ __forceinline__ Cols<V> load_cols(const float* __restrict__ p) {
  static_assert(V == 1 || V == 2, "columns a lane");
  Cols<V> c;
  if (V == 2) {
    const float2 x = __ldcg(reinterpret_cast<const float2*>(p));
    c.v[0] = x.x; c.v[V - 1] = x.y;
  } else {
    c.v[0] = __ldcg(p);
  }
  return c;
}
template <int V, int NP> struct Partials { Cols<V> c[NP]; };
template <int V, int NP>
__device__ __forceinline__ void issue_partials(Partials<V, NP>& x, const float* __restrict__ p, size_t stride, int i0, int S) {
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    if (i0 + j < S) x.c[j] = load_cols<V>(p + (size_t)(i0 + j) * stride);
    else
#pragma unroll
      for (int k = 0; k < V; ++k) x.c[j].v[k] = 0.f;
  }
}
template <int V, int NP>
__device__ __forceinline__ void add_partials(const Partials<V, NP>& x, float* s) {
#pragma unroll
  for (int j = 0; j < NP; ++j)
#pragma unroll
    for (int k = 0; k < V; ++k) s[k] += x.c[j].v[k];
}
// the partials from index i0 on
template <int V>
__device__ __forceinline__ void sum_partials_from(const float* __restrict__ p, size_t stride, int i0, int S, float* s) {
  for (; i0 < S; i0 += 8) {
    Partials<V, 8> x;
    issue_partials(x, p, stride, i0, S);
    add_partials(x, s);
  }
}

// QKV finalisation: sum the split-K partials, apply the folded norm factor and the bias, rotate q and k
// (rotate-half pairs j, j + D/2), write q to its buffer and k, v into the layer's cache planes.  One warp per (row, head), D / 64
// pairs a lane, four warps a CTA: a grid that is resident at once beside the GEMM CTAs which already hold their shared memory
// (with one CTA of two warps per (row, head) it took two waves: 3.7 us a layer of the 3B shape and 32 rows).
template <typename T, int D>
__global__ void __launch_bounds__(128) fin_qkv_kernel(const float* __restrict__ part, int S, int m, const float2* __restrict__ cs,
                                                      const float* __restrict__ ssq, int nt, float inv_h, float eps,
                                                      const float* __restrict__ bq, const float* __restrict__ bk, const float* __restrict__ bv,
                                                      const float* __restrict__ sq, const float* __restrict__ sk, const float* __restrict__ sv,
                                                      T* __restrict__ q, T* __restrict__ kc, T* __restrict__ vc, int pos0, int hq, int hkv,
                                                      int max_seq, const int* __restrict__ len_ptr, const float* __restrict__ x_scale,
                                                      float* __restrict__ amax_zero, KStamp* stamp) {
  constexpr int HALF = D / 2, V = D / 64;
  if (threadIdx.x == 0) stamp_start(stamp);
  pdl_trigger();
  const int heads = hq + 2 * hkv, unit = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int r = unit / heads, head = unit - r * heads, j = lane * V;
  const bool live = r < m;
  // not written by any kernel of this forward: the cache length word, the scales and the biases
  if (len_ptr) pos0 = *len_ptr;
  const int kind = head < hq ? 0 : (head < hq + hkv ? 1 : 2), hl = head - (kind == 0 ? 0 : (kind == 1 ? hq : hq + hkv));
  float sc[2][V], bi[2][V];
  {
    const float* scp = kind == 0 ? sq : (kind == 1 ? sk : sv);
    const float* bip = kind == 0 ? bq : (kind == 1 ? bk : bv);
#pragma unroll
    for (int i = 0; i < 2 * V; ++i) {
      const int c = hl * D + (i / V) * HALF + j + i % V;
      sc[i / V][i % V] = live && scp ? scp[c] : 1.f;      // fp8 weights: per-output-channel factors
      bi[i / V][i % V] = live && bip ? bip[c] : 0.f;
    }
  }
  pdl_wait();
  if (threadIdx.x == 0) stamp_released(stamp);
  if (!live) return;
  // W8A8: the row's slot of the running maximum that this layer's gate/up epilogue raises; its last reader (the
  // quantisation in front of the previous layer's down projection) is long done, its next writers start after this kernel
  if (amax_zero && head == 0 && lane == 0) amax_zero[r] = 0.f;
  // every load of this kernel is issued before the first result is needed
  const int width = heads * D;
  const size_t sstride = (size_t)m * width;
  const float* pa = part + (size_t)r * width + head * D + j;
  float ssq_v = 0.f;
  for (int t = lane; t < nt; t += 32) ssq_v += __ldcg(ssq + (size_t)r * nt + t);
  const float xs = x_scale ? __ldcg(x_scale + r) : 1.f;     // W8A8: the partial sums are sums of code products; the row's factor joins the norm's
  float2 c[V];
#pragma unroll
  for (int k = 0; k < V; ++k) c[k] = kind < 2 ? __ldcg(&cs[r * HALF + j + k]) : make_float2(1.f, 0.f);
  Partials<V, 16> va, vb;
  issue_partials(va, pa, sstride, 0, S);
  issue_partials(vb, pa + HALF, sstride, 0, S);
  const float rstd = rsqrtf(warp_sum(ssq_v) * inv_h + eps) * xs;
  float a[V], b[V];
#pragma unroll
  for (int k = 0; k < V; ++k) a[k] = b[k] = 0.f;
  add_partials(va, a);
  add_partials(vb, b);
  sum_partials_from<V>(pa, sstride, 16, S, a);
  sum_partials_from<V>(pa + HALF, sstride, 16, S, b);
  T oa[V], ob[V];
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const float x = a[k] * rstd * sc[0][k] + bi[0][k], y = b[k] * rstd * sc[1][k] + bi[1][k];
    oa[k] = from_f32<T>(kind < 2 ? x * c[k].x - y * c[k].y : x);
    ob[k] = from_f32<T>(kind < 2 ? y * c[k].x + x * c[k].y : y);
  }
  T* o = kind == 0 ? q + ((size_t)r * hq + head) * D : (kind == 1 ? kc : vc) + ((size_t)hl * max_seq + pos0 + r) * D;
  if (V == 2) {
    *reinterpret_cast<uint32_t*>(o + j) = *reinterpret_cast<const uint32_t*>(oa);
    *reinterpret_cast<uint32_t*>(o + j + HALF) = *reinterpret_cast<const uint32_t*>(ob);
  } else {
    o[j] = oa[0];
    o[j + HALF] = ob[0];
  }
  if (threadIdx.x == 0) stamp_end(stamp, true);
}
void launch_fin_qkv(const float* part, int S, int m, const float* cs, const float* ssq, int nt, int hidden, float eps,
                    const float* bq, const float* bk, const float* bv, const float* sq, const float* sk, const float* sv, void* q, void* kc, void* vc, int pos0, int hq,
                    int hkv, int d, int max_seq, int kv_type, cudaStream_t st, const int* len_ptr, KStamp* stamp, const float* x_scale,
                    float* amax_zero) {
  auto go = [&](auto kern, auto* qt, auto* kt, auto* vt) {
    launch_pdl(kern, dim3(ceil_div(m * (hq + 2 * hkv), 4)), dim3(128), 0, st, part, S, m, (const float2*)cs, ssq, nt, 1.f / (float)hidden,
               eps, bq, bk, bv, sq, sk, sv, qt, kt, vt, pos0, hq, hkv, max_seq, len_ptr, x_scale, amax_zero, stamp);
  };
  if (kv_type == KV_F16) {
    if (d == 128) go(fin_qkv_kernel<__half, 128>, (__half*)q, (__half*)kc, (__half*)vc);
    else go(fin_qkv_kernel<__half, 64>, (__half*)q, (__half*)kc, (__half*)vc);
  } else {
    if (d == 128) go(fin_qkv_kernel<bf16, 128>, (bf16*)q, (bf16*)kc, (bf16*)vc);
    else go(fin_qkv_kernel<bf16, 64>, (bf16*)q, (bf16*)kc, (bf16*)vc);
  }
}

// Residual finalisation: h += sum of split-K partials; xg = h * gain of the next norm (stored as `fmt`);
// ssq[row][tile] = sum of h^2 over the tile's 128 columns (hidden even).  Two warps per (row, tile), two columns a lane, two such
// pairs a CTA, all partials in flight at once (a CTA of four warps per (row, tile), one column a thread: 12.2 us for a layer's two launches of the 7B
// shape at 64 rows, 8.6 now, 8.4 : 7.1 at 32 rows; four columns a lane: the partials no longer fit and 64 rows of the 3B shape took 9.4 instead of 8.7).
__global__ void __launch_bounds__(128) fin_resid_kernel(const float* __restrict__ part, int S, int m, int hidden,
                                                        float* __restrict__ h, const float* __restrict__ g,
                                                        void* __restrict__ xg, size_t lo_off, int fmt, float* __restrict__ ssq, int nt,
                                                        const float* __restrict__ scale, const float* __restrict__ x_scale,
                                                        float* __restrict__ amax_out, KStamp* stamp) {
  if (threadIdx.x == 0) stamp_start(stamp);
  pdl_trigger();
  const int pair = threadIdx.x >> 6, unit = blockIdx.x * 2 + pair;
  const int r = unit / nt, t = unit - r * nt, c = t * 128 + (threadIdx.x & 63) * 2;
  const bool in = r < m && c < hidden;
  // weights (gain, scale) do not depend on the predecessor
  const float g0 = in ? g[c] : 0.f, g1 = in ? g[c + 1] : 0.f;
  float s0 = in && scale ? scale[c] : 1.f, s1 = in && scale ? scale[c + 1] : 1.f;
  pdl_wait();
  if (threadIdx.x == 0) stamp_released(stamp);
  float ss = 0.f, am = 0.f;
  if (in) {
    const size_t idx = (size_t)r * hidden + c, sstride = (size_t)m * hidden;
    Partials<2, 18> pv;
    issue_partials(pv, part + idx, sstride, 0, S);
    const Cols<2> hv = load_cols<2>(h + idx);
    if (x_scale) {     // W8A8: the partial sums are sums of code products
      const float xs = __ldcg(x_scale + r);
      s0 *= xs;
      s1 *= xs;
    }
    float s[2] = {0.f, 0.f};
    add_partials(pv, s);
    sum_partials_from<2>(part + idx, sstride, 18, S, s);
    const float x0 = hv.v[0] + s[0] * s0, x1 = hv.v[1] + s[1] * s1, a0 = x0 * g0, a1 = x1 * g1;
    *reinterpret_cast<float2*>(h + idx) = make_float2(x0, x1);
    store_act2(xg, lo_off, idx, a0, a1, fmt);
    ss = fmaf(x0, x0, x1 * x1);
    if (amax_out) am = fmaxf(abs_as_f16(a0), abs_as_f16(a1));
  }
  // the tile's sum of squares and (W8A8: the next projection's quantiser) the maximum of the stored xg
  __shared__ float red_s[4], red_m[4];
  ss = warp_sum(ss);
  if (amax_out) am = warp_max(am);
  if ((threadIdx.x & 31) == 0) { red_s[threadIdx.x >> 5] = ss; red_m[threadIdx.x >> 5] = am; }
  __syncthreads();
  if ((threadIdx.x & 63) == 0 && r < m) {
    ssq[(size_t)r * nt + t] = red_s[2 * pair] + red_s[2 * pair + 1];
    if (amax_out) amax_out[(size_t)r * nt + t] = fmaxf(red_m[2 * pair], red_m[2 * pair + 1]);
    if (threadIdx.x == 0) stamp_end(stamp, true);
  }
}
// The same for the many rows of a prompt (hidden a multiple of 4, no W8A8): one warp per (row, tile of 128 columns), four
// columns per lane.  Bound by the bytes it moves; the kernel above, whose CTAs exist to have every load of a few rows in
// flight at once, took 35 us for 1024 x 2048 with two splits.
__global__ void __launch_bounds__(256) fin_resid_rows_kernel(const float* __restrict__ part, int S, int m, int hidden,
                                                             float* __restrict__ h, const float* __restrict__ g, void* __restrict__ xg,
                                                             size_t lo_off, int fmt, float* __restrict__ ssq, int nt,
                                                             const float* __restrict__ scale, KStamp* stamp) {
  if (threadIdx.x == 0) stamp_start(stamp);
  pdl_trigger();
  const int idx_w = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int r = idx_w / nt, t = idx_w - r * nt, c = t * 128 + lane * 4;
  pdl_wait();
  if (threadIdx.x == 0) stamp_released(stamp);
  if (r >= m) return;
  float ss = 0.f;
  if (c < hidden) {
    const size_t idx = (size_t)r * hidden + c, sstride = (size_t)m * hidden;
    const float4 hv = *reinterpret_cast<const float4*>(h + idx);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < S; s0 += 4) {
      float4 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        v[j] = (s0 + j < S) ? __ldcs(reinterpret_cast<const float4*>(part + idx + (size_t)(s0 + j) * sstride)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int j = 0; j < 4; ++j) { a.x += v[j].x; a.y += v[j].y; a.z += v[j].z; a.w += v[j].w; }
    }
    float x[4] = {a.x, a.y, a.z, a.w};
    const float hh[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      x[e] = hh[e] + x[e] * (scale ? scale[c + e] : 1.f);
      ss = fmaf(x[e], x[e], ss);
    }
    *reinterpret_cast<float4*>(h + idx) = make_float4(x[0], x[1], x[2], x[3]);
    store_act4(xg, lo_off, idx, make_float4(x[0] * g[c], x[1] * g[c + 1], x[2] * g[c + 2], x[3] * g[c + 3]), fmt);
  }
  ss = warp_sum(ss);
  if (lane == 0) ssq[(size_t)r * nt + t] = ss;
  if (threadIdx.x == 0) stamp_end(stamp, true);
}
void launch_fin_resid_rows(const float* part, int S, int m, int hidden, float* h, const float* g, void* xg, size_t lo_off, int fmt,
                           float* ssq, int nt, const float* scale, cudaStream_t st, KStamp* stamp) {
  launch_pdl(fin_resid_rows_kernel, dim3((m * nt + 7) / 8), dim3(256), 0, st, part, S, m, hidden, h, g, xg, lo_off, fmt, ssq, nt, scale, stamp);
}
void launch_fin_resid(const float* part, int S, int m, int hidden, float* h, const float* g, void* xg, size_t lo_off, int fmt,
                      float* ssq, int nt, const float* scale, cudaStream_t st, KStamp* stamp, const float* x_scale, float* amax_out) {
  launch_pdl(fin_resid_kernel, dim3(ceil_div(m * nt, 2)), dim3(128), 0, st, part, S, m, hidden, h, g, xg, lo_off, fmt, ssq, nt, scale, x_scale,
             amax_out, stamp);
}

// Merge the per-warp softmax statistics of the LM-head epilogue into confidence and prediction per row.
// stats[e * m + row] = (max, sum exp(l - max), argmax id) for e in [0, n_part).  grid m rows, 256 threads.
__global__ void __launch_bounds__(512) stats_merge_kernel(const float4* __restrict__ stats, int n_part, int m,
                                                          float* __restrict__ conf, int32_t* __restrict__ pred, KStamp* stamp) {
  if (threadIdx.x == 0) stamp_start(stamp);
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) stamp_released(stamp);
  __shared__ float sm_m[16], sm_s[16];
  __shared__ int sm_i[16];
  const int r = blockIdx.x;
  float mx = -INFINITY, s = 0.f;
  int ix = 0x7fffffff;
  auto merge = [&](float m2, float s2, int i2) {
    if (s2 == 0.f) return;
    if (s == 0.f) { mx = m2; s = s2; ix = i2; return; }
    const float mn = fmaxf(mx, m2);
    s = s * __expf(mx - mn) + s2 * __expf(m2 - mn);
    if (m2 > mx || (m2 == mx && i2 < ix)) ix = i2;
    mx = mn;
  };
  // ten loads in flight per thread: at the 3B / 7B vocabularies (4.7k partials per row) one L2 round trip in all
  for (int e0 = threadIdx.x; e0 < n_part; e0 += 10 * blockDim.x) {
    float4 v[10];
#pragma unroll
    for (int j = 0; j < 10; ++j) {
      const int e = e0 + j * blockDim.x;
      v[j] = e < n_part ? __ldcg(&stats[(size_t)e * m + r]) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int j = 0; j < 10; ++j) merge(v[j].x, v[j].y, __float_as_int(v[j].z));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, mx, o), s2 = __shfl_xor_sync(0xffffffffu, s, o);
    const int i2 = __shfl_xor_sync(0xffffffffu, ix, o);
    merge(m2, s2, i2);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) { sm_m[w] = mx; sm_s[w] = s; sm_i[w] = ix; }
  __syncthreads();
  if (threadIdx.x == 0) {
    mx = sm_m[0]; s = sm_s[0]; ix = sm_i[0];
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k) merge(sm_m[k], sm_s[k], sm_i[k]);
    conf[r] = 1.f / s;
    pred[r] = ix;
    stamp_end(stamp);
  }
}
void launch_stats_merge(const void* stats, int n_part, int m, float* conf, int32_t* pred, cudaStream_t st, KStamp* stamp) {
  launch_pdl(stats_merge_kernel, dim3(m), dim3(512), 0, st, (const float4*)stats, n_part, m, conf, pred, stamp);
}

// ================================================================================================
// unmask selection (one CTA of 64 threads; n <= 64)
// ================================================================================================
__global__ void select_kernel(const float* __restrict__ conf, const int32_t* __restrict__ pred,
                              int32_t* __restrict__ tokens, uint8_t* __restrict__ masked,
                              uint8_t* __restrict__ unmask, int32_t* __restrict__ info, int n, int rule,
                              float threshold, int k, int shift, cudaGraphConditionalHandle cond, int loop,
                              const StepDev* __restrict__ dev) {
  pdl_trigger();
  pdl_wait();
  if (dev) { rule = dev->rule; threshold = dev->threshold; k = dev->k; shift = dev->shift; }
  __shared__ float c[64];
  __shared__ int mk[64];
  int i = threadIdx.x;
  // shift = 1: position i is predicted by row i - 1; position 0 has no predictor and is never selected
  c[i] = (i < n && i >= shift) ? conf[i - shift] : -1.f;
  mk[i] = (i < n && i >= shift) ? (int)masked[i] : 0;
  // a masked position 0 under shift = 1 has no predictor: nothing is revealed and it is reported as remaining
  const int stuck = (shift && n > 0 && masked[0]) ? 1 : 0;
  __syncthreads();
  int is_m = mk[i];
  int rank = 0, n_masked = 0;
  for (int j = 0; j < n; ++j) {
    if (!mk[j]) continue;
    ++n_masked;
    if (c[j] > c[i] || (c[j] == c[i] && j < i)) ++rank;
  }
  int sel;
  if (rule == 0) {
    int hit = is_m && (c[i] > threshold);
    int any = __syncthreads_or(hit);
    sel = any ? hit : (is_m && rank == 0);
  } else {
    sel = is_m && rank < k;
  }
  if (stuck) sel = 0;
  int n_sel = __syncthreads_count(sel);
  if (i < n) {
    unmask[i] = (uint8_t)sel;
    if (sel) { tokens[i] = pred[i - shift]; masked[i] = 0; }
  }
  if (i == 0) {
    const int left = n_masked - n_sel + stuck;
    info[0] = n_sel; info[1] = left; info[2] = info[2] + 1;
    if (loop) {
      // body of the on-device decode loop: run another denoise step while masked positions are left.  Every step
      // reveals at least one position, so the loop ends after at most n steps; the explicit count is a second bound.
      const int it = info[5] + 1;
      info[5] = it;
      cudaGraphSetConditional(cond, (left > 0 && n_sel > 0 && it < n) ? 1u : 0u);
    }
  }
}
void launch_select(const float* conf, const int32_t* pred, int32_t* tokens, uint8_t* masked, uint8_t* unmask,
                   int32_t* info, int n, int rule, float threshold, int k, cudaStream_t st, int shift,
                   cudaGraphConditionalHandle cond, int loop) {
  select_kernel<<<1, 64, 0, st>>>(conf, pred, tokens, masked, unmask, info, n, rule, threshold, k, shift, cond, loop, nullptr);
}
void launch_select_dev(const float* conf, const int32_t* pred, int32_t* tokens, uint8_t* masked, uint8_t* unmask, int32_t* info, int n,
                       const StepDev* dev, cudaStream_t st) {
  launch_pdl(select_kernel, dim3(1), dim3(64), 0, st, conf, pred, tokens, masked, unmask, info, n, 0, 0.f, 0, 0, (cudaGraphConditionalHandle)0, 0, dev);
}
__global__ void set_step_kernel(StepDev* dev, StepDev v) { *dev = v; }
void launch_set_step(StepDev* dev, StepDev v, cudaStream_t st) { set_step_kernel<<<1, 1, 0, st>>>(dev, v); }

// Longest accepted prefix of a drafted block d against the causal predictions a (a[j] predicts the token after d[j]):
// k = 1 + (first j in [0, n-2] with a[j] != d[j+1]; n-1 if none).  out = {k, a[k-1]}.
__global__ void accept_kernel(const int32_t* __restrict__ a, const int32_t* __restrict__ d, int n, int32_t* __restrict__ out) {
  __shared__ int first;
  if (threadIdx.x == 0) first = n - 1;
  __syncthreads();
  const int j = threadIdx.x;
  if (j < n - 1 && a[j] != d[j + 1]) atomicMin(&first, j);
  __syncthreads();
  if (threadIdx.x == 0) { out[0] = first + 1; out[1] = a[first]; }
}
void launch_accept(const int32_t* a, const int32_t* d, int n, int32_t* out, cudaStream_t st) {
  accept_kernel<<<1, 64, 0, st>>>(a, d, n, out);
}

// Read-only streaming of a buffer: every CTA walks its share with 16-byte loads, eight in flight per thread, and folds
// what it reads into one word (so that the loads cannot be dropped).  A yardstick for the read bandwidth a kernel of this
// library can reach at all; no part of the decoding path.
__global__ void __launch_bounds__(256) stream_read_kernel(const uint4* __restrict__ buf, size_t n16, unsigned* __restrict__ sink) {
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned acc = 0;
  for (; i + 7 * stride < n16; i += 8 * stride) {
    uint4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = __ldcs(buf + i + u * stride);
#pragma unroll
    for (int u = 0; u < 8; ++u) acc ^= v[u].x ^ v[u].y ^ v[u].z ^ v[u].w;
  }
  for (; i < n16; i += stride) { const uint4 v = __ldcs(buf + i); acc ^= v.x ^ v.y ^ v.z ^ v.w; }
  if (acc == 0x9e3779b9u) atomicAdd(sink, 1u);     // practically never: keeps the loads alive without a store per thread
}
void launch_stream_read(const void* buf, size_t bytes, unsigned* sink, int ctas, cudaStream_t st) {
  stream_read_kernel<<<ctas, 256, 0, st>>>((const uint4*)buf, bytes / 16, sink);
}

// ---- quadratic self-speculative decoding (Appendix B, Alg. 2) --------------------------------------------------------
// Row order of the B (B + 1) rows of one forward: rows 0 .. B-1 are the draft tokens d_0 .. d_{B-1} (the first tokens of
// the groups), row B + i B + (j - 1) is mask token j (1 <= j <= B) of group i.  With the first tokens in front, the rows
// whose K / V outlive the forward ("keep every (B+1)-th entry", and of those the accepted ones) are the first k staging
// rows of the cache.
//   pos_off[r]: position id minus the position of d_0: i for a first token, i + j for a mask token
//   mask[r]   : bit r' = row r reads row r'.  (b) first token i reads first tokens <= i; (c) a mask token of group i reads
//               its group's first token and all its mask tokens; (d) nothing else -- chain != 0: also the first tokens of
//               the groups before i.
__global__ void quad_layout_kernel(int B, int chain, unsigned long long* __restrict__ mask, int* __restrict__ pos_off) {
  const int r = threadIdx.x, n = B * (B + 1);
  if (r >= n) return;
  if (r < B) {
    mask[r] = (2ull << r) - 1ull;                              // bits 0 .. r
    pos_off[r] = r;
  } else {
    const int i = (r - B) / B, j = (r - B) % B + 1;
    const unsigned long long group = ((B == 64 ? 0ull : (1ull << B)) - 1ull) << (B + i * B);   // its B mask rows
    unsigned long long m = group | (1ull << i);
    if (chain) m |= (1ull << i) - 1ull;
    mask[r] = m;
    pos_off[r] = i + j;
  }
}
void launch_quad_layout(int B, int chain, unsigned long long* mask, int* pos_off, cudaStream_t st) {
  quad_layout_kernel<<<1, 64, 0, st>>>(B, chain, mask, pos_off);
}
// tokens of the rows above from the draft d
__global__ void quad_build_kernel(const int32_t* __restrict__ d, int B, int mask_id, int32_t* __restrict__ tokens,
                                  uint8_t* __restrict__ masked) {
  const int r = threadIdx.x;
  if (r >= B * (B + 1)) return;
  tokens[r] = r < B ? d[r] : mask_id;
  masked[r] = r >= B;
}
void launch_quad_build(const int32_t* d, int B, int mask_id, int32_t* tokens, uint8_t* masked, cudaStream_t st) {
  quad_build_kernel<<<1, 64, 0, st>>>(d, B, mask_id, tokens, masked);
}
// Alg. 2 step 1: d_0 = the token the prompt's last row predicts, d_i = prediction of mask row i - 1 (shift by one)
__global__ void quad_first_draft_kernel(const int32_t* __restrict__ pred, int32_t first, int B, int32_t* __restrict__ d) {
  const int i = threadIdx.x;
  if (i < B) d[i] = i == 0 ? first : pred[i - 1];
}
void launch_quad_first_draft(const int32_t* pred, int32_t first, int B, int32_t* d, cudaStream_t st) {
  quad_first_draft_kernel<<<1, 64, 0, st>>>(pred, first, B, d);
}
// Alg. 2's verify loop on the predictions of one forward (P_{i,0} = pred[i], P_{i,j} = pred[B + i B + j - 1]):
// k = 1; while k < B and P_{k-1,0} = d_k: k += 1.  accepted[0 .. k) = d_0 .. d_{k-1}; d <- P_{k-1,1..B}; out = {k}.
__global__ void quad_accept_kernel(const int32_t* __restrict__ pred, int32_t* __restrict__ d, int B, int32_t* __restrict__ accepted,
                                   int32_t* __restrict__ out) {
  __shared__ int k_s;
  __shared__ int32_t old_d[64];
  const int t = threadIdx.x;
  if (t < B) old_d[t] = d[t];
  __syncthreads();
  if (t == 0) {
    int k = 1;
    while (k < B && pred[k - 1] == old_d[k]) ++k;
    k_s = k;
    out[0] = k;
  }
  __syncthreads();
  const int k = k_s;
  if (t < B) {
    if (accepted) accepted[t] = t < k ? old_d[t] : -1;
    d[t] = pred[B + (k - 1) * B + t];
  }
}
void launch_quad_accept(const int32_t* pred, int32_t* d, int B, int32_t* accepted, int32_t* out, cudaStream_t st) {
  quad_accept_kernel<<<1, 64, 0, st>>>(pred, d, B, accepted, out);
}

// Commit of the finished block (Bc rows) and opening of the next one (Bn rows) for ONE forward over Bc + Bn rows:
// rows = [finished tokens ; next block's initial tokens]; mask: a finished row reads the finished rows up to itself
// (Alg. 1 verify mask), a row of the next block reads every row (the committed block is part of its context, its own
// block is bidirectional); the block state becomes the next block's.
__global__ void fuse_begin_kernel(int32_t* __restrict__ blk_tokens, uint8_t* __restrict__ blk_masked, int Bc,
                                  const int32_t* __restrict__ init, int Bn, int mask_id, int32_t* __restrict__ rows,
                                  unsigned long long* __restrict__ mask, int32_t* __restrict__ info) {
  __shared__ int32_t nxt[64];
  const int i = threadIdx.x, n = Bc + Bn;
  const int32_t old = i < Bc ? blk_tokens[i] : 0;
  nxt[i] = (i < Bn && init) ? init[i] : mask_id;
  __syncthreads();
  if (i < n) {
    rows[i] = i < Bc ? old : nxt[i - Bc];
    mask[i] = i < Bc ? (2ull << i) - 1ull : (n == 64 ? ~0ull : (1ull << n) - 1ull);
  }
  const int m = (i < Bn) && (nxt[i] == mask_id);
  if (i < Bn) { blk_tokens[i] = nxt[i]; blk_masked[i] = (uint8_t)m; }
  const int cnt = __syncthreads_count(m);
  if (i == 0) { info[0] = 0; info[1] = cnt; info[2] = 0; }
}
void launch_fuse_begin(int32_t* blk_tokens, uint8_t* blk_masked, int Bc, const int32_t* init, int Bn, int mask_id, int32_t* rows,
                       unsigned long long* mask, int32_t* info, cudaStream_t st) {
  fuse_begin_kernel<<<1, 64, 0, st>>>(blk_tokens, blk_masked, Bc, init, Bn, mask_id, rows, mask, info);
}

__global__ void init_block_kernel(int32_t* tokens, uint8_t* masked, int32_t* info, const int32_t* init, int n, int mask_id,
                                  int step) {
  int i = threadIdx.x;
  int t = (i < n && init) ? init[i] : mask_id;
  int m = (i < n) && (t == mask_id);
  if (i < n) { tokens[i] = t; masked[i] = (uint8_t)m; }
  int cnt = __syncthreads_count(m);
  if (i == 0) { info[0] = 0; info[1] = cnt; info[2] = step; }
}
void launch_init_block(int32_t* tokens, uint8_t* masked, int32_t* info, const int32_t* init, int n, int mask_id, int step,
                       cudaStream_t st) {
  init_block_kernel<<<1, 64, 0, st>>>(tokens, masked, info, init, n, mask_id, step);
}

}  // namespace fdk
