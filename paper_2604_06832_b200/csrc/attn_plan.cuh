// What the attention kernels of the decode and the prompt path share.
#pragma once
#include "tc_ptx.cuh"

namespace fdk {

constexpr int AT_KEYS = 128;   // keys per shared-memory tile
constexpr float LOG2E = 1.4426950408889634f;

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Split of T keys into chunks of whole AT_KEYS-key tiles, at most `bound` chunks (the same on host and device, so a launch
// whose grid was sized for `bound` can take the sequence length from device memory).
__host__ __device__ inline void attn_chunking(int T, int bound, int* chunk_keys, int* n_chunks) {
  const int tiles = (T + AT_KEYS - 1) / AT_KEYS;
  int want = bound < tiles ? bound : tiles;
  if (want < 1) want = 1;
  *chunk_keys = ((tiles + want - 1) / want) * AT_KEYS;
  *n_chunks = (T + *chunk_keys - 1) / *chunk_keys;
}

template <typename T> __device__ __forceinline__ uint32_t pack2(float lo, float hi);
template <> __device__ __forceinline__ uint32_t pack2<bf16>(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
template <> __device__ __forceinline__ uint32_t pack2<__half>(float lo, float hi) {
  __half2 v = __floats2half2_rn(lo, hi);       // probabilities lie in [0, 1]: no range concern
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ float ex2(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// two fp32 operations in one instruction
__device__ __forceinline__ float2 fma2(const float2& a, const float2& b, const float2& c) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
      "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 add2(const float2& a, const float2& b) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tadd.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}

// ---- steps of the online softmax, one thread per row, 64 scores ------------------------------------------------
__device__ __forceinline__ float row_max64(const float* s) {
  float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
  for (int c = 0; c < 64; c += 8)
#pragma unroll
    for (int k = 0; k < 4; ++k) mx[k] = fmaxf(fmaxf(mx[k], s[c + k]), s[c + 4 + k]);
  return fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
}
// P = 2^(s sl2 - ref) as 16-bit values into the columns of S at tensor-memory address ts; returns the row's sum
template <typename E>
__device__ __forceinline__ float exp_pack64(const float* s, float sl2, float ref, uint32_t ts) {
  float2 sum[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  const float2 sl = make_float2(sl2, sl2), mr = make_float2(-ref, -ref);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t pk[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      float2 e = fma2(make_float2(s[h * 32 + 2 * c], s[h * 32 + 2 * c + 1]), sl, mr);
      e = make_float2(ex2(e.x), ex2(e.y));
      sum[c & 1] = add2(sum[c & 1], e);
      pk[c] = pack2<E>(e.x, e.y);
    }
    tmem_st16(ts + h * 16, pk);
  }
  return (sum[0].x + sum[0].y) + (sum[1].x + sum[1].y);
}
// the row's accumulator (D columns at `to`) times f
template <int D>
__device__ __forceinline__ void scale_acc(uint32_t to, float f) {
#pragma unroll 1
  for (int c = 0; c < D; c += 16) {
    float o[16];
    tmem_ld16(to + c, o);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < 16; ++k) o[k] *= f;
    tmem_st16(to + c, reinterpret_cast<const uint32_t*>(o));
  }
}

}  // namespace fdk
