// Launchers of the fdvlm kernels (host-callable; all asynchronous on `st`).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "common.cuh"

namespace fdk {

// ---- small-M linear: y[m,n] = sum_k x[m,k] w[n,k] (* scale[n]) (+ bias[n]) ---------------------
struct LinearArgs {
  const void* x;        // [m, k]   fp32 (DT_F32) or bf16
  const void* w;        // [n, k]   per dtype
  const float* scale;   // [n] or null
  const float* bias;    // [n] or null
  float* y;             // [m, n] fp32 result
  int m, n, k;
  int dtype;            // DT_*
  void* workspace;      // split-K partial sums
  size_t workspace_bytes;
};

// ---- elementwise / reduction kernels -----------------------------------------------------------
// tokens outside [0, vocab) read row 0 and leave ST_BAD_TOKEN in *status
// One launch for an fp32 row block: embedding gather and rotary table (as launch_rope_table).
void launch_embed_rope_f32(const void* table, const int32_t* tokens, float* h, int n, int hidden, int vocab, int* status, float* cs,
                           int pos0, int head_dim, float theta, const int* len_ptr, const int* pos_off, cudaStream_t st);
void launch_embed_f32(const void* table, const int32_t* tokens, float* h, int n, int hidden, int vocab, int* status, cudaStream_t st);
void launch_bf16_to_e5m2x3(const void* in, void* out, size_t n, cudaStream_t st);       // planes n bytes apart
// W8A8: rows of k f16 values (k a multiple of 8) -> e4m3 codes and scale[row] = max / 448, from amax[row][n_amax], partial maxima
// of |value| left by whoever wrote the rows; and bf16 rows -> f16 (saturating) -> the same, maxima included.
void launch_quantize_rows(const void* x, int m, int k, const float* amax, int n_amax, void* codes, float* scale, cudaStream_t st);
void launch_quantize_bf16_rows(const void* in, int m, int k, void* codes, float* scale, cudaStream_t st);
void launch_rope_table(float* cs, int n, int pos0, int head_dim, float theta, cudaStream_t st, const int* len_ptr = nullptr,
                       KStamp* stamp = nullptr, const int* pos_off = nullptr);
// quadratic self-speculative decoding (Appendix B, Alg. 2): row layout, input tokens, first draft, verify loop
// read-only streaming yardstick (see the kernel)
void launch_stream_read(const void* buf, size_t bytes, unsigned* sink, int ctas, cudaStream_t st);
// commit of the finished block + opening of the next one as one forward: rows, row masks, block state
void launch_fuse_begin(int32_t* blk_tokens, uint8_t* blk_masked, int Bc, const int32_t* init, int Bn, int mask_id, int32_t* rows,
                       unsigned long long* mask, int32_t* info, cudaStream_t st);
void launch_quad_layout(int B, int chain, unsigned long long* mask, int* pos_off, cudaStream_t st);
void launch_quad_build(const int32_t* d, int B, int mask_id, int32_t* tokens, uint8_t* masked, cudaStream_t st);
void launch_quad_first_draft(const int32_t* pred, int32_t first, int B, int32_t* d, cudaStream_t st);
void launch_quad_accept(const int32_t* pred, int32_t* d, int B, int32_t* accepted, int32_t* out, cudaStream_t st);
void launch_set_len(int* len_ptr, int value, cudaStream_t st);
// Unmask selection + block-state update.  info = {n_unmasked, n_remaining, step_index}.
// loop = 1: the launch is the last node of a conditional WHILE body; it counts the iteration in info[5] and sets `cond`
// to "masked positions remain".
void launch_select(const float* conf, const int32_t* pred, int32_t* tokens, uint8_t* masked, uint8_t* unmask,
                   int32_t* info, int n, int rule, float threshold, int k, cudaStream_t st, int shift = 0,
                   cudaGraphConditionalHandle cond = 0, int loop = 0);
// dev: the parameters come from device memory (a captured launch).
struct StepDev { int rule; float threshold; int k, shift; };
void launch_set_step(StepDev* dev, StepDev v, cudaStream_t st);
void launch_select_dev(const float* conf, const int32_t* pred, int32_t* tokens, uint8_t* masked, uint8_t* unmask, int32_t* info, int n,
                       const StepDev* dev, cudaStream_t st);
// out[0] = accepted length k, out[1] = a[k - 1] (Alg. 1 "Accept: left-to-right comparison")
void launch_accept(const int32_t* a, const int32_t* d, int n, int32_t* out, cudaStream_t st);
void launch_init_block(int32_t* tokens, uint8_t* masked, int32_t* info, const int32_t* init, int n, int mask_id,
                       int step, cudaStream_t st);

// ---- the exact fp32 path (exact_f32.cu) ---------------------------------------------------------------
// One projection over m rows x [m, k], with the RMSNorm in front of it (gain set) and what follows it:
//   QKV   : w = q, k, v; bias, rotary (cs); q rows into out, K / V rows into the cache planes kc, vc at pos0 (*len_ptr)
//   RESID : out [m, n0] += x w^T
//   SWIGLU: w = gate, up; out [m, n0] = silu(gate) * up
//   LOGITS: out [m, n0] (nullable); stats[tile][m] (nullable): as TcOut's, f32_logit_tiles entries
enum { FL_QKV = 0, FL_RESID = 1, FL_SWIGLU = 2, FL_LOGITS = 3 };
struct F32Linear {
  int mode, m, k;
  const float* x;
  const float* gain; float inv_h, eps;
  const float *w[3], *bias[3]; int n[3];
  float *out, *kc, *vc;
  const float* cs; const int* len_ptr; int pos0, hq, hkv, d, max_seq;
  float4* stats; int mask_id;
};
int f32_logit_tiles(int vocab, int m);      // entries of `stats` for each of m rows, at most ceil(vocab / 16)
cudaError_t launch_linear_f32(const F32Linear& p, cudaStream_t st);

// ---- tensor-core (tcgen05 + TMA) small-M GEMM, bf16 ---------------------------------------------------
enum { TC_MODE_PARTIAL = 0, TC_MODE_SWIGLU = 1, TC_MODE_LOGITS = 2 };
// Up to three bf16 matrices that share x and K; their outputs sit side by side in one row of width ld.
struct TcGroup {
  const void* x; int m, k;   // bf16 weights: bf16 rows (hi plane); fp8 weights: XF_E5M2X3 rows (first plane); a8: rows of e4m3 codes
  const void* x_lo;          // bf16 weights, nullable: the rows' low-order bf16 plane (x = hi + lo); fp8 weights: second plane
  const void* x_3;           // fp8 weights: third plane
  const void* w[3]; int n[3]; int n_mats;
  const float* scale[3];
  int fp8;   // weights are e4m3 bytes (scale[] holds the per-output-channel factors)
  int a8;    // with fp8: the rows are e4m3 codes, one factor per row (W8A8); PARTIAL and SWIGLU only
};
// What the GEMM leaves behind.
//   PARTIAL: part[split][m][ld] = split-K partial sums (*splits_out of them) for the caller's reduce kernel
//   SWIGLU : act[m][n0] = silu(x w0^T * rstd * s0) * (x w1^T * rstd * s1)   (w[0] = gate, w[1] = up)
//   LOGITS : y[m][ld] = (x w^T) * rstd[row] * scale (when write_logits), and stats[tile * 4 + quarter][m] = (max, sum exp(l - max), argmax id)
//            over the 32 vocabulary ids a warp holds, mask_id excluded
// rstd[row] = rsqrt(sum_t ssq_in[row][t] / hidden + eps) when ssq_in is set (RMSNorm folded into the consumer), else 1.
struct TcOut {
  int mode;
  float* part; size_t part_bytes; int* splits_out;
  float* y; int ld;
  void* act; size_t act_lo_off; int act_fmt;   // SWIGLU output, stored as XF_* (lo plane act_lo_off elements on)
  const float* ssq_in; int nt_in; int hidden; float eps;
  void* stats; int mask_id; int write_logits;
  int* status;   // two device words: [0] set non-zero if a bounded wait inside the kernel gave up; [1] read at kernel
                 // start, non-zero sends every role down its give-up path at once
  KStamp* stamp; // in-chain timing of the launch, nullable
  // a8 groups: x_scale[row] = the factor of the row's codes.  The accumulators are sums of code products: PARTIAL output still
  // lacks the factor (the reduce kernel applies it), SWIGLU applies it itself and raises amax_out[row] (atomic maximum: zero
  // before the launch) to max |act[row]|.
  const float* x_scale;
  float* amax_out;
};
// Tensor map of a 2-D row-major [rows, cols] tensor with box {64 columns, box_rows}, zero fill outside the tensor
// (cached per argument set).  kind TM_BF16 / TM_F16: 16-bit elements, 128-byte swizzle; TM_E4M3: bytes, no swizzle;
// TM_E4M3_128: bytes, box of 128 columns, 128-byte swizzle.  False when the driver entry point is missing or the encode fails.
enum { TM_BF16 = 0, TM_E4M3 = 1, TM_F16 = 2, TM_E4M3_128 = 3 };
bool make_tmap(CUtensorMap* tm, const void* ptr, int rows, int cols, int box_rows, int kind = TM_BF16);
// The planes of a GEMM input, equally far apart, as one 3-D tensor [planes, rows, cols]: one box fetches a k-block of all of them.
bool make_tmap_planes(CUtensorMap* tm, const void* ptr, int rows, int cols, int planes, size_t plane_bytes, int box_rows, int kind);
bool tc_linear_supported(int m, int n, int k, int dtype);
// Split-K workspace of a group with m rows, output width ld, `tiles` 128-row weight tiles and depth k.
size_t tc_workspace_bytes(int m, int ld, int tiles, int k);
// The decode path's gate / up projection (SWIGLU): one equal share of the features per SM (gemm_gu.cu).  next (nullable): the weights
// [next_n, next_k], of the same type, that the following launch streams.  Groups that are not supported go to tc_group_launch.
bool gemm_gu_supported(const TcGroup& g);
cudaError_t gemm_gu_launch(const TcGroup& g, const TcOut& o, const void* next, int next_n, int next_k, cudaStream_t st);
cudaError_t tc_group_launch(const TcGroup& g, const TcOut& o, cudaStream_t st);

// SM count of the current device (cached per device: one process may drive several GPUs).
int sm_count();

// ---- large-M GEMM of the prompt path (prefill_gemm.cu) ---------------------------------------------------------
//   QKV    : w = q, k, v; out = q rows [m][n0] after bias and rotary (cs), K / V into the cache planes kc, vc at pos0
//   RESID  : h += x w^T * scale; out = h * gain (XF_*, lo plane out_lo_off on); ssq_out[row][nt] = sums of h^2 per 128 columns
//   SWIGLU : w = gate, up; out[m][n0] = silu(gate) * up
//   PARTIAL: part[splits][m][n0] = split-K partial sums, left to fin_resid
// The folded norm factor comes from ssq_in as in TcOut.  fp8: e4m3 weights and f16 rows; else bf16 weights and hi / lo planes.
enum { PF_QKV = 0, PF_RESID = 1, PF_SWIGLU = 2, PF_PARTIAL = 3 };
struct PfGemm {
  int mode, m, k, x_rows, fp8, n_mats;        // x_rows >= m: rows that x holds
  const void *x, *x_lo;
  const void* w[3]; int n[3];
  const float *scale[3], *bias[3];
  const float* ssq_in; int nt; float inv_h, eps;
  void* out; size_t out_lo_off; int out_fmt;
  void *kc, *vc; const float* cs; int pos0, max_seq, d, kv_type;
  float* h; const float* gain; float* ssq_out;
  float* part; int splits;
  unsigned* arrived;      // nullable: sm_count() * 4 zeroed words; with `part` (256 x 256 sums per two SMs) tiles may come in pieces
  int* status;
  KStamp* stamp;          // in-chain timing of the launch, nullable
};
int prefill_splits(int m, int n, int k);
cudaError_t prefill_gemm_launch(const PfGemm& g, cudaStream_t st);

// Tensor-core path glue.  ssq[row][nt] holds per-128-column partial sums of h^2; xg / lo_off / fmt: a GEMM input
// stored as XF_* (common.cuh).  q, kc, vc of fin_qkv are KV_BF16 or KV_F16 elements (kv_type).
void launch_embed_prep(const void* table, const int32_t* tokens, const void* rows, float* h, void* xg, size_t lo_off, int fmt,
                       const float* g, float* ssq, int nt, int n, int hidden, int vocab, int* status, cudaStream_t st,
                       KStamp* stamp = nullptr, float* amax = nullptr);
void launch_fin_qkv(const float* part, int S, int m, const float* cs, const float* ssq, int nt, int hidden, float eps,
                    const float* bq, const float* bk, const float* bv, const float* sq, const float* sk, const float* sv, void* q,
                    void* kc, void* vc, int pos0, int hq,
                    int hkv, int d, int max_seq, int kv_type, cudaStream_t st, const int* len_ptr = nullptr, KStamp* stamp = nullptr,
                    const float* x_scale = nullptr, float* amax_zero = nullptr);
void launch_fin_resid(const float* part, int S, int m, int hidden, float* h, const float* g, void* xg, size_t lo_off, int fmt,
                      float* ssq, int nt, const float* scale, cudaStream_t st, KStamp* stamp = nullptr,
                      const float* x_scale = nullptr, float* amax_out = nullptr);
void launch_fin_resid_rows(const float* part, int S, int m, int hidden, float* h, const float* g, void* xg, size_t lo_off, int fmt,
                           float* ssq, int nt, const float* scale, cudaStream_t st, KStamp* stamp = nullptr);
void launch_stats_merge(const void* stats, int n_part, int m, float* conf, int32_t* pred, cudaStream_t st, KStamp* stamp = nullptr);

// ---- attention -----------------------------------------------------------------------------------
struct AttnArgs {
  const void* q;   // [n, Hq, d]
  const void* kc;  // [Hkv, max_seq, d]
  const void* vc;
  void* out;       // [n, Hq*d]
  int n, cache_len, max_seq, hq, hkv, d, causal, dtype;
  int kv_type;          // tensor-core kernel: element type of q, kc, vc (KV_BF16 / KV_F16)
  int out_fmt;          // tensor-core kernel: storage of `out` (XF_*), lo plane out_lo_off elements on
  size_t out_lo_off;
  const unsigned long long* row_mask;   // nullable, n <= 64 words: bit r' of word r = row r reads row r' of this forward
                                        // (the cached keys are always read); overrides `causal`
  void* workspace;
  const int* len_ptr;   // nullable: device word holding the cache length (overrides cache_len)
  int* status;          // nullable: device status words (see TcOut::status)
  float* amax_out;      // nullable (tensor-core kernel): [n][hq] maxima of |out| as stored, per row and head
  // tensor-core kernel, nullable: matrices [next_n, next_k] (bf16 or e4m3) of a launch that follows soon, every third pair of k-blocks of which is asked for in L2, by CTAs on every SM
  const void* next_w[2]; int next_n, next_k, next_fp8;
  KStamp* stamp;        // nullable: decode: two consecutive entries (attention, chunk merge); prompt path: one
};
// Prompt path: causal attention of any number of rows, one CTA per (256 rows, query head), no key split (prefill_attn.cu).
cudaError_t launch_prefill_attention(const AttnArgs& a, cudaStream_t st);
size_t attention_workspace_bytes(int n, int hq, int hkv, int d);

}  // namespace fdk
