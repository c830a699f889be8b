// The decoder forward of one step as a launch sequence (Fast-dVLM Sec. 3.4; Appendix B Alg. 1 for the
// two attention modes), in two flavours: the exact CUDA-core path (fp32 weights) and the tensor-core path (bf16 and fp8
// weights).
#include "handle.h"

namespace fdk {

int launch_linear_simt(const LinearArgs& a, cudaStream_t st, cudaError_t* err);
size_t simt_workspace_bytes(int m, int n, int k);
int launch_attention_f32(const AttnArgs& a, cudaStream_t st, cudaError_t* err);
size_t attention_tc_workspace_bytes(int n, int hq, int hkv, int d);
int launch_attention_tc(const AttnArgs& a, cudaStream_t st, cudaError_t* err);
void launch_splitk_epilogue(const float* part, int S, int m, int n, const float* scale, const float* bias, float* y,
                            cudaStream_t st, const float* x_scale = nullptr);

thread_local char g_create_error[512] = "";

// Stand-alone projection.  The caller's workspace starts with OP_HEAD bytes for the two status words (see
// TcOut::status; cleared here on the stream), then -- fp8 weights only -- the bf16 rows as XF_E5M2X3 planes (W8A8: as e4m3
// codes, followed by one 256-byte-rounded array of per-row factors), then the split-K partial sums.
static size_t op_scale_bytes(int m, int dtype) { return dtype == DT_A8 ? (((size_t)m * 4 + 255) / 256) * 256 : 0; }
static size_t op_x16_bytes(int m, int k, int dtype, int fp8_row_bytes = 3) {
  if (dtype == DT_FP8) return (((size_t)m * k * fp8_row_bytes + 255) / 256) * 256;
  return dtype == DT_A8 ? (((size_t)m * k + 255) / 256) * 256 + op_scale_bytes(m, dtype) : 0;
}
size_t linear_workspace_bytes(int m, int n, int k, int dtype, int fp8_row_bytes) {
  const int wdt = dtype == DT_A8 ? DT_FP8 : dtype;
  size_t a = dtype == DT_A8 ? 0 : simt_workspace_bytes(m, n, k);
  size_t b = tc_linear_supported(m, n, k, wdt) ? tc_workspace_bytes(m, n, (n + 127) / 128, k) + op_x16_bytes(m, k, dtype, fp8_row_bytes) : 0;
  return OP_HEAD + (a > b ? a : b);
}

// One projection y = x w^T (* scale) (+ bias) (+ y): bf16 / fp8 weights go to the tensor-core kernel
// (split-K partial sums + fixed-order reduction), everything else to the CUDA-core kernel.
int launch_linear(const LinearArgs& a, cudaStream_t st, cudaError_t* err) {
  if (!a.workspace || a.workspace_bytes < OP_HEAD) { *err = cudaErrorInvalidValue; return -1; }
  *err = cudaMemsetAsync(a.workspace, 0, 8, st);
  if (*err != cudaSuccess) return -1;
  LinearArgs b = a;
  b.workspace = (char*)a.workspace + OP_HEAD;
  b.workspace_bytes = a.workspace_bytes - OP_HEAD;
  const bool a8 = a.dtype == DT_A8;
  if (!tc_linear_supported(a.m, a.n, a.k, a8 ? DT_FP8 : a.dtype)) {
    if (a8) { *err = cudaErrorNotSupported; return -1; }      // the quantising projection exists on the tensor cores only
    return launch_linear_simt(b, st, err);
  }
  TcGroup g;
  memset(&g, 0, sizeof(g));
  g.x = a.x; g.m = a.m; g.k = a.k; g.w[0] = a.w; g.n[0] = a.n; g.n_mats = 1;
  g.fp8 = (a.dtype == DT_FP8 || a8); g.a8 = a8;
  const size_t x16 = op_x16_bytes(a.m, a.k, a.dtype);
  if (b.workspace_bytes < x16) { *err = cudaErrorInvalidValue; return -1; }
  float* x_scale = a8 ? (float*)((char*)b.workspace + x16 - op_scale_bytes(a.m, a.dtype)) : nullptr;
  int launched = 2;
  if (a8) {
    launch_quantize_bf16_rows(a.x, a.m, a.k, b.workspace, x_scale, st);
    g.x = b.workspace;
    ++launched;
  } else if (g.fp8) {
    const size_t plane = (size_t)a.m * a.k;
    launch_bf16_to_e5m2x3(a.x, b.workspace, plane, st);
    g.x = b.workspace; g.x_lo = (const char*)g.x + plane; g.x_3 = (const char*)g.x + 2 * plane;
    ++launched;
  }
  float* part = (float*)((char*)b.workspace + x16);
  int splits = 0;
  TcOut o;
  memset(&o, 0, sizeof(o));
  o.mode = TC_MODE_PARTIAL; o.part = part; o.part_bytes = b.workspace_bytes - x16; o.splits_out = &splits;
  o.ld = a.n; o.status = (int*)a.workspace;
  *err = tc_group_launch(g, o, st);
  if (*err != cudaSuccess) return -1;
  launch_splitk_epilogue(part, splits, a.m, a.n, a.scale, a.bias, a.y, st, x_scale);
  *err = cudaGetLastError();
  return *err == cudaSuccess ? launched : -1;
}

size_t attention_workspace_bytes(int n, int hq, int hkv, int d) { return attention_tc_workspace_bytes(n, hq, hkv, d); }
// 16-bit rows go to the split-KV tensor-core kernel, fp32 rows to the exact CUDA-core kernel.
int launch_attention(const AttnArgs& a, cudaStream_t st, cudaError_t* err) {
  return a.dtype == DT_F32 ? launch_attention_f32(a, st, err) : launch_attention_tc(a, st, err);
}

int stage_rows(fdvlm_t* h, int row0, int n, const int32_t* tokens, const void* embeds, int mode, const int* len_ptr) {
  const int H = h->cfg.hidden;
  if (h->use_tc) {
    launch_embed_prep(h->w.embed, tokens, embeds, h->h + (size_t)row0 * H, (char*)h->a + (size_t)row0 * H * xf_bytes(h->xfmt), h->a_lo, h->xfmt,
                      h->layers[0].g_attn, h->ssq + (size_t)row0 * h->nt, h->nt, n, H, h->cfg.vocab, h->info + 3, h->st, nullptr,
                      h->act8 ? h->amax_a + (size_t)row0 * h->nt : nullptr);
  } else if (tokens && mode >= 0) {
    launch_embed_rope_f32(h->w.embed, tokens, h->h + (size_t)row0 * H, n, H, h->cfg.vocab, h->info + 3, h->cs, h->cache_len, h->cfg.head_dim,
                          h->cfg.rope_theta, len_ptr, mode == MODE_MASKED ? h->q_pos_off : nullptr, h->st);
  } else {
    launch_embed_f32(tokens ? h->w.embed : embeds, tokens, h->h + (size_t)row0 * H, n, H, h->cfg.vocab, h->info + 3, h->st);
  }
  h->launches++;
  CU(h, cudaGetLastError());
  return FDVLM_OK;
}

// The rows of a group: a GEMM input stored as `fmt`, planes lo_off elements apart, from element row0_elems on.
static void set_rows(TcGroup* g, const void* x, size_t lo_off, size_t row0_elems, int fmt) {
  const char* p = (const char*)x + row0_elems * xf_bytes(fmt);
  g->x = p;
  g->x_lo = (fmt == XF_BF16X2 || fmt == XF_E5M2X3) ? p + lo_off * xf_bytes(fmt) : nullptr;
  g->x_3 = fmt == XF_E5M2X3 ? p + 2 * lo_off : nullptr;
  g->fp8 = fmt == XF_E5M2X3 || fmt == XF_F16;
}
int stage_prefill_rows(fdvlm_t* h, int row0, int n, const int32_t* tokens, const void* embeds) {
  const size_t H = h->cfg.hidden;
  launch_embed_prep(h->w.embed, tokens, embeds, h->pf_h + row0 * H, (char*)h->pf_a + row0 * H * 2, h->pf_rows * H, h->pf_fmt,
                    h->layers[0].g_attn, h->pf_ssq + (size_t)row0 * h->nt, h->nt, n, (int)H, h->cfg.vocab, h->info + 3, h->st);
  h->launches++;
  CU(h, cudaGetLastError());
  return FDVLM_OK;
}

// In-chain timing: the record of the next launch, null while it is off.
static KStamp* next_stamp(fdvlm_t* h, bool stamped, int kind) {
  if (!stamped || h->stamp_used >= FDVLM_MAX_STAMPS) return nullptr;
  h->stamp_kind.push_back(kind);
  return h->stamps + h->stamp_used++;
}

// ---- prompt path ---------------------------------------------------------------------------------------------------------
// per layer: [QKV GEMM + norm factor, bias, rotary, K/V rows] [causal attention] [O GEMM + residual, gain, ssq]
//            [gate/up GEMM + SwiGLU] [down GEMM + residual, gain, ssq]
// O and down of a short prompt: split-K partial sums + fin_resid_rows (see prefill_splits).
int forward_prefill(fdvlm_t* h, int n, int want_last_logits) {
  const fdvlm_config& c = h->cfg;
  const int H = c.hidden, I = c.intermediate, d = c.head_dim, nt = h->nt;
  const int NQ = c.n_q_heads * d, NKV = c.n_kv_heads * d;
  const size_t R = h->pf_rows;
  const bool fp8 = h->dt == DT_FP8, stamped = h->prof_on == 2;
  cudaError_t e = cudaSuccess;
  if (stamped) {
    h->stamp_kind.clear();
    h->stamp_used = 0;
    CU(h, cudaMemsetAsync(h->stamps, 0xFF, sizeof(KStamp) * FDVLM_MAX_STAMPS, h->st));
  }
  auto gemm = [&](int mode, int kind, const void* x, size_t ld, int k) {
    PfGemm g;
    memset(&g, 0, sizeof(g));
    g.mode = mode; g.m = n; g.k = k; g.x_rows = (int)R; g.fp8 = fp8; g.n_mats = 1;
    g.x = x; g.x_lo = fp8 ? nullptr : (const char*)x + R * ld * 2;
    g.nt = nt; g.inv_h = 1.f / (float)H; g.eps = c.rms_eps; g.status = h->info + 3;
    g.part = h->pf_part; g.arrived = h->pf_arrived; g.stamp = next_stamp(h, stamped, kind);
    return g;
  };
  auto run = [&](const PfGemm& g) {
    prof_begin(h, 0);
    e = prefill_gemm_launch(g, h->st);
    prof_end(h);
    h->launches++;
    return e == cudaSuccess;
  };
  // residual add of x w^T, the next norm's gain and sums of squares
  auto resid = [&](int kind, const void* x, size_t ld, int k, const void* w, const float* scale, const float* gain, int fmt) {
    PfGemm g = gemm(PF_RESID, kind, x, ld, k);
    g.w[0] = w; g.n[0] = H;
    g.splits = prefill_splits(n, H, k);
    if (g.splits > 1 && (size_t)g.splits * n * H * sizeof(float) <= h->pf_part_bytes) {
      g.mode = PF_PARTIAL;
      if (!run(g)) return false;
      launch_fin_resid_rows(h->pf_part, g.splits, n, H, h->pf_h, gain, h->pf_a, R * H, fmt, h->pf_ssq, nt, scale, h->st,
                            next_stamp(h, stamped, FDVLM_K_FIN_RESID));
      h->launches++;
      return true;
    }
    g.scale[0] = scale; g.h = h->pf_h; g.gain = gain; g.out = h->pf_a; g.out_lo_off = R * H; g.out_fmt = fmt; g.ssq_out = h->pf_ssq;
    return run(g);
  };
  // (a forward whose waits gave up may have left some)
  CU(h, cudaMemsetAsync(h->pf_arrived, 0, (size_t)sm_count() * 4 * sizeof(unsigned), h->st));
  launch_rope_table(h->pf_cs, n, h->cache_len, d, c.rope_theta, h->st, nullptr, next_stamp(h, stamped, FDVLM_K_ROPE_TABLE));
  h->launches++;
  for (int l = 0; l < c.n_layers; ++l) {
    const fdvlm_layer_weights& lw = h->layers[l];
    PfGemm g = gemm(PF_QKV, FDVLM_K_GEMM_QKV, h->pf_a, H, H);
    g.n_mats = 3;
    g.w[0] = lw.wq; g.w[1] = lw.wk; g.w[2] = lw.wv; g.n[0] = NQ; g.n[1] = g.n[2] = NKV;
    g.scale[0] = lw.s_q; g.scale[1] = lw.s_k; g.scale[2] = lw.s_v; g.bias[0] = lw.bq; g.bias[1] = lw.bk; g.bias[2] = lw.bv;
    g.ssq_in = h->pf_ssq; g.out = h->pf_q; g.kc = kv_ptr(h, l, 0); g.vc = kv_ptr(h, l, 1); g.cs = h->pf_cs;
    g.pos0 = h->cache_len; g.max_seq = c.max_seq; g.d = d; g.kv_type = h->kv_type;
    if (!run(g)) return fail(h, FDVLM_ERR_CUDA, "qkv projection launch: %s", cudaGetErrorString(e));
    AttnArgs at;
    memset(&at, 0, sizeof(at));
    at.q = h->pf_q; at.kc = kv_ptr(h, l, 0); at.vc = kv_ptr(h, l, 1); at.out = h->pf_ao; at.n = n; at.cache_len = h->cache_len;
    at.max_seq = c.max_seq; at.hq = c.n_q_heads; at.hkv = c.n_kv_heads; at.d = d; at.causal = 1; at.kv_type = h->kv_type;
    at.out_fmt = h->pf_fmt; at.out_lo_off = R * NQ; at.status = h->info + 3;
    at.stamp = next_stamp(h, stamped, FDVLM_K_ATTENTION);
    prof_begin(h, 1);
    e = launch_prefill_attention(at, h->st);
    prof_end(h);
    h->launches++;
    if (e != cudaSuccess) return fail(h, FDVLM_ERR_CUDA, "attention launch: %s", cudaGetErrorString(e));
    if (!resid(FDVLM_K_GEMM_O, h->pf_ao, NQ, NQ, lw.wo, lw.s_o, lw.g_mlp, h->pf_fmt))
      return fail(h, FDVLM_ERR_CUDA, "o projection launch: %s", cudaGetErrorString(e));
    g = gemm(PF_SWIGLU, FDVLM_K_GEMM_GATE_UP, h->pf_a, H, H);
    g.n_mats = 2;
    g.w[0] = lw.w_gate; g.w[1] = lw.w_up; g.n[0] = g.n[1] = I; g.scale[0] = lw.s_gate; g.scale[1] = lw.s_up;
    g.ssq_in = h->pf_ssq; g.out = h->pf_act; g.out_lo_off = R * I; g.out_fmt = h->pf_fmt;
    if (!run(g)) return fail(h, FDVLM_ERR_CUDA, "gate/up projection launch: %s", cudaGetErrorString(e));
    const bool last = l + 1 == c.n_layers;
    if (!resid(FDVLM_K_GEMM_DOWN, h->pf_act, I, I, lw.w_down, lw.s_down, last ? h->w.g_final : h->layers[l + 1].g_attn, last ? h->head_fmt : h->pf_fmt))
      return fail(h, FDVLM_ERR_CUDA, "down projection launch: %s", cudaGetErrorString(e));
  }
  if (want_last_logits) {
    TcOut o;
    memset(&o, 0, sizeof(o));
    o.mode = TC_MODE_LOGITS; o.status = h->info + 3; o.y = h->logits; o.ld = c.vocab; o.write_logits = 1;
    o.stamp = next_stamp(h, stamped, FDVLM_K_GEMM_LM_HEAD);
    o.ssq_in = h->pf_ssq + (size_t)(n - 1) * nt; o.nt_in = nt; o.hidden = H; o.eps = c.rms_eps; o.stats = h->stats; o.mask_id = c.mask_id;
    TcGroup lm;
    memset(&lm, 0, sizeof(lm));
    lm.m = 1; lm.k = H; lm.n_mats = 1; lm.n[0] = c.vocab;
    lm.w[0] = c.tie_embeddings ? h->w.embed : h->w.lm_head;
    set_rows(&lm, h->pf_a, R * H, (size_t)(n - 1) * H, h->head_fmt);
    if (!c.tie_embeddings) lm.scale[0] = h->w.s_lm_head;
    prof_begin(h, 0);
    e = tc_group_launch(lm, o, h->st);
    prof_end(h);
    h->launches++;
    if (e != cudaSuccess) return fail(h, FDVLM_ERR_CUDA, "lm head launch: %s", cudaGetErrorString(e));
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return fail(h, FDVLM_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(e));
  return FDVLM_OK;
}

// ---- exact fp32 path ----------------------------------------------------------------------------------
// per layer: [norm + QKV, bias, rotary, K/V rows] [attention] [O + residual] [norm + gate/up + SwiGLU] [down + residual]
static int forward_rows_f32(fdvlm_t* h, int n, int mode, int logits_rows, int want_logits, const int* len_ptr, bool rope_done) {
  const fdvlm_config& c = h->cfg;
  const int H = c.hidden, I = c.intermediate, d = c.head_dim, NQ = c.n_q_heads * d, NKV = c.n_kv_heads * d;
  cudaError_t e = cudaSuccess;
  auto lin = [&](int lm, const void* x, int m, int k, const float* gain, const void* w, int nn, float* out) {
    F32Linear g;
    memset(&g, 0, sizeof(g));
    g.mode = lm; g.x = (const float*)x; g.m = m; g.k = k; g.gain = gain; g.inv_h = 1.f / (float)H; g.eps = c.rms_eps;
    g.w[0] = (const float*)w; g.n[0] = nn; g.out = out;
    return g;
  };
  auto run = [&](const F32Linear& g) {
    prof_begin(h, 0);
    e = launch_linear_f32(g, h->st);
    prof_end(h);
    h->launches++;
    return e == cudaSuccess;
  };
  if (!rope_done) {
    launch_rope_table(h->cs, n, h->cache_len, d, c.rope_theta, h->st, len_ptr, nullptr, mode == MODE_MASKED ? h->q_pos_off : nullptr);
    h->launches++;
  }
  for (int l = 0; l < c.n_layers; ++l) {
    const fdvlm_layer_weights& lw = h->layers[l];
    F32Linear g = lin(FL_QKV, h->h, n, H, lw.g_attn, lw.wq, NQ, (float*)h->q);
    g.w[1] = (const float*)lw.wk; g.w[2] = (const float*)lw.wv; g.n[1] = g.n[2] = NKV;
    g.bias[0] = lw.bq; g.bias[1] = lw.bk; g.bias[2] = lw.bv;
    g.kc = (float*)kv_ptr(h, l, 0); g.vc = (float*)kv_ptr(h, l, 1); g.cs = h->cs; g.len_ptr = len_ptr; g.pos0 = h->cache_len;
    g.hq = c.n_q_heads; g.hkv = c.n_kv_heads; g.d = d; g.max_seq = c.max_seq;
    if (!run(g)) return fail(h, FDVLM_ERR_CUDA, "qkv projection launch: %s", cudaGetErrorString(e));
    AttnArgs at;
    memset(&at, 0, sizeof(at));
    at.q = h->q; at.kc = kv_ptr(h, l, 0); at.vc = kv_ptr(h, l, 1); at.out = h->ao; at.n = n; at.cache_len = h->cache_len; at.len_ptr = len_ptr;
    at.max_seq = c.max_seq; at.hq = c.n_q_heads; at.hkv = c.n_kv_heads; at.d = d; at.causal = (mode == MODE_CAUSAL); at.dtype = DT_F32;
    at.row_mask = (mode == MODE_MASKED) ? h->q_mask : (mode == MODE_FUSED ? h->f_mask : nullptr);
    prof_begin(h, 1);
    const int r = launch_attention(at, h->st, &e);
    prof_end(h);
    if (r < 0) return fail(h, FDVLM_ERR_CUDA, "attention launch: %s", cudaGetErrorString(e));
    h->launches += r;
    if (!run(lin(FL_RESID, h->ao, n, NQ, nullptr, lw.wo, H, h->h)))
      return fail(h, FDVLM_ERR_CUDA, "o projection launch: %s", cudaGetErrorString(e));
    g = lin(FL_SWIGLU, h->h, n, H, lw.g_mlp, lw.w_gate, I, (float*)h->act);
    g.w[1] = (const float*)lw.w_up; g.n[1] = I;
    if (!run(g)) return fail(h, FDVLM_ERR_CUDA, "gate/up projection launch: %s", cudaGetErrorString(e));
    if (!run(lin(FL_RESID, h->act, n, I, nullptr, lw.w_down, H, h->h)))
      return fail(h, FDVLM_ERR_CUDA, "down projection launch: %s", cudaGetErrorString(e));
  }
  if (logits_rows > 0) {
    const bool all = logits_rows == n;
    const int first = all ? 0 : n - 1;
    F32Linear g = lin(FL_LOGITS, h->h + (size_t)first * H, n - first, H, h->w.g_final, c.tie_embeddings ? h->w.embed : h->w.lm_head, c.vocab,
                      (!all || want_logits) ? h->logits : nullptr);
    g.stats = all ? (float4*)h->stats : nullptr; g.mask_id = c.mask_id;
    if (!run(g)) return fail(h, FDVLM_ERR_CUDA, "lm head launch: %s", cudaGetErrorString(e));
    if (all) {
      launch_stats_merge(h->stats, f32_logit_tiles(c.vocab, n), n, h->conf, h->pred, h->st);
      h->launches++;
    }
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return fail(h, FDVLM_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(e));
  return FDVLM_OK;
}

// ---- tensor-core path (bf16 / fp8 weights) ---------------------------------------------------------------
// per layer: [QKV GEMM -> split-K partials] [sum + folded norm + bias + rotary + K/V staging] [attention + chunk merge]
//            [O GEMM -> partials] [sum + residual + gain + ssq] [gate/up GEMM, folded norm + SwiGLU epilogue]
//            [down GEMM -> partials] [sum + residual + gain + ssq]
// head:      [LM-head GEMM, folded final norm, logits + softmax statistics epilogue] [statistics merge]
// stamped: every launch gets the next record of h->stamps (in-chain timing, fdvlm_profile_enable(h, 2)).
static int forward_rows_tc(fdvlm_t* h, int n, int mode, int logits_rows, int want_logits, const int* len_ptr, bool stamped) {
  const fdvlm_config& c = h->cfg;
  const int H = c.hidden, I = c.intermediate, d = c.head_dim, nt = h->nt;
  const int NQ = c.n_q_heads * d, NKV = c.n_kv_heads * d, NQKV = NQ + 2 * NKV;
  float* part = (float*)h->ws;
  cudaError_t e = cudaSuccess;
  if (stamped) { h->stamp_kind.clear(); h->stamp_used = 0; }
  auto stamp = [&](int kind) { return next_stamp(h, stamped, kind); };
  const bool a8 = h->act8 != 0;                      // W8A8: the four layer projections quantise their input rows
  // a GEMM input buffer: hi (or only) plane, and its lo plane when the format has one
  auto group = [&](const void* x, size_t lo_off, size_t row0_elems, int m, int k, int nm, const void* w0, int n0, const void* w1, int n1,
                   const void* w2, int n2) {
    TcGroup g;
    memset(&g, 0, sizeof(g));
    set_rows(&g, x, lo_off, row0_elems, h->xfmt);
    g.m = m; g.k = k; g.n_mats = nm;
    g.w[0] = w0; g.n[0] = n0; g.w[1] = w1; g.n[1] = n1; g.w[2] = w2; g.n[2] = n2;
    return g;
  };
  // W8A8: a projection's input rows as e4m3 codes, from the partial maxima that whoever wrote them left
  const float* xs = a8 ? h->xscale : nullptr;
  auto quantised = [&](TcGroup g, const float* amax, int n_amax) {
    if (!a8) return g;
    launch_quantize_rows(g.x, g.m, g.k, amax, n_amax, h->codes, h->xscale, h->st);
    h->launches++;
    g.x = h->codes; g.x_lo = g.x_3 = nullptr; g.a8 = 1;
    return g;
  };
  auto out = [&](int tc_mode, int kind) {
    TcOut o;
    memset(&o, 0, sizeof(o));
    o.mode = tc_mode; o.status = h->info + 3; o.part = part; o.part_bytes = h->ws_bytes; o.stamp = stamp(kind);
    return o;
  };
  auto gemm = [&](const TcGroup& g, const TcOut& o) {
    prof_begin(h, 0);
    e = tc_group_launch(g, o, h->st);
    prof_end(h);
    h->launches++;
    return e == cudaSuccess;
  };
  launch_rope_table(h->cs, n, h->cache_len, d, c.rope_theta, h->st, len_ptr, stamp(FDVLM_K_ROPE_TABLE),
                    mode == MODE_MASKED ? h->q_pos_off : nullptr);
  h->launches++;
  for (int l = 0; l < c.n_layers; ++l) {
    const fdvlm_layer_weights& lw = h->layers[l];
    int S = 0;
    TcOut o = out(TC_MODE_PARTIAL, FDVLM_K_GEMM_QKV);
    o.ld = NQKV; o.splits_out = &S;
    if (!gemm(quantised(group(h->a, h->a_lo, 0, n, H, 3, lw.wq, NQ, lw.wk, NKV, lw.wv, NKV), h->amax_a, nt), o))
      return fail(h, FDVLM_ERR_CUDA, "qkv projection launch: %s", cudaGetErrorString(e));
    launch_fin_qkv(part, S, n, h->cs, h->ssq, nt, H, c.rms_eps, lw.bq, lw.bk, lw.bv, lw.s_q, lw.s_k, lw.s_v, h->q, kv_ptr(h, l, 0), kv_ptr(h, l, 1),
                   h->cache_len, c.n_q_heads, c.n_kv_heads, d, c.max_seq, h->kv_type, h->st, len_ptr, stamp(FDVLM_K_FIN_QKV),
                   xs, a8 ? h->amax_act : nullptr);
    AttnArgs at;
    memset(&at, 0, sizeof(at));
    at.len_ptr = len_ptr;
    at.q = h->q; at.kc = kv_ptr(h, l, 0); at.vc = kv_ptr(h, l, 1); at.out = h->ao; at.n = n; at.cache_len = h->cache_len;
    at.max_seq = c.max_seq; at.hq = c.n_q_heads; at.hkv = c.n_kv_heads; at.d = d; at.causal = (mode == MODE_CAUSAL);
    at.row_mask = (mode == MODE_MASKED) ? h->q_mask : (mode == MODE_FUSED ? h->f_mask : nullptr);
    at.dtype = h->dt; at.workspace = h->ws; at.kv_type = h->kv_type; at.out_fmt = h->xfmt; at.out_lo_off = h->ao_lo;
    at.status = h->info + 3;
    // Memory idles from here to the gate / up projection: part of its weights is brought into L2 meanwhile (NextWeights, every third pair).
    // Not with fp8 weights from 33 rows on, where gate / up is bound by its MMAs (three planes) and not by its weights.
    // us a step without : with, a process each: 3B shape, 12 layers: 4 rows 687 : 672, 32 rows 762 : 739, 64 rows 862 : 842.  7B shape, 8 layers,
    // fp8: 8 rows 608 : 597, 32 rows 658 : 647, 33 rows 682 : 685, 36 rows 686 : 691, 40 rows 697 : 705, 64 rows 855 : 867;
    // W8A8 (one plane): 8 rows 652 : 633, 32 rows 721 : 697, 33 rows 719 : 706, 41 rows 724 : 718, 48 rows 725 : 722, 64 rows 804 : 798.
    if (h->dt == DT_BF16 || a8 || n <= 32) {
      at.next_w[0] = lw.w_gate; at.next_w[1] = lw.w_up; at.next_n = I; at.next_k = H; at.next_fp8 = h->dt == DT_FP8;
    }
    at.amax_out = a8 ? h->amax_ao : nullptr;
    at.stamp = stamp(FDVLM_K_ATTENTION);
    if (at.stamp && !stamp(FDVLM_K_ATTN_MERGE)) at.stamp = nullptr;     // the launcher uses two consecutive records
    prof_begin(h, 1);
    int r = launch_attention(at, h->st, &e);
    prof_end(h);
    if (r < 0) return fail(h, FDVLM_ERR_CUDA, "attention launch: %s", cudaGetErrorString(e));
    h->launches += r + 1;
    o = out(TC_MODE_PARTIAL, FDVLM_K_GEMM_O);
    o.ld = H; o.splits_out = &S;
    if (!gemm(quantised(group(h->ao, h->ao_lo, 0, n, NQ, 1, lw.wo, H, nullptr, 0, nullptr, 0), h->amax_ao, c.n_q_heads), o))
      return fail(h, FDVLM_ERR_CUDA, "o projection launch: %s", cudaGetErrorString(e));
    launch_fin_resid(part, S, n, H, h->h, lw.g_mlp, h->a, h->a_lo, h->xfmt, h->ssq, nt, lw.s_o, h->st, stamp(FDVLM_K_FIN_RESID),
                     xs, a8 ? h->amax_a : nullptr);
    o = out(TC_MODE_SWIGLU, FDVLM_K_GEMM_GATE_UP);
    o.act = h->act; o.act_lo_off = h->act_lo; o.act_fmt = h->xfmt;
    o.ssq_in = h->ssq; o.nt_in = nt; o.hidden = H; o.eps = c.rms_eps;
    o.x_scale = xs; o.amax_out = a8 ? h->amax_act : nullptr;
    TcGroup gu = group(h->a, h->a_lo, 0, n, H, 2, lw.w_gate, I, lw.w_up, I, nullptr, 0);
    gu.scale[0] = lw.s_gate; gu.scale[1] = lw.s_up;
    gu = quantised(gu, h->amax_a, nt);
    prof_begin(h, 0);
    e = gemm_gu_supported(gu) ? gemm_gu_launch(gu, o, lw.w_down, H, I, h->st) : tc_group_launch(gu, o, h->st);
    prof_end(h);
    h->launches++;
    if (e != cudaSuccess)
      return fail(h, FDVLM_ERR_CUDA, "gate/up projection launch: %s", cudaGetErrorString(e));
    o = out(TC_MODE_PARTIAL, FDVLM_K_GEMM_DOWN);
    o.ld = H; o.splits_out = &S;
    if (!gemm(quantised(group(h->act, h->act_lo, 0, n, I, 1, lw.w_down, H, nullptr, 0, nullptr, 0), h->amax_act, 1), o))
      return fail(h, FDVLM_ERR_CUDA, "down projection launch: %s", cudaGetErrorString(e));
    // the last layer feeds the LM head, whose table (a tied bf16 embedding under fp8 layer weights) may want another format
    const bool last = (l + 1 == c.n_layers);
    const float* g_next = last ? h->w.g_final : h->layers[l + 1].g_attn;
    launch_fin_resid(part, S, n, H, h->h, g_next, h->a, h->a_lo, last ? h->head_fmt : h->xfmt, h->ssq, nt, lw.s_down, h->st,
                     stamp(FDVLM_K_FIN_RESID), xs, (a8 && !last) ? h->amax_a : nullptr);
    h->launches += 2;
  }
  if (logits_rows > 0) {
    const int first = (logits_rows == n) ? 0 : n - 1;
    const int m = n - first;
    const void* table = c.tie_embeddings ? h->w.embed : h->w.lm_head;
    TcOut o = out(TC_MODE_LOGITS, FDVLM_K_GEMM_LM_HEAD);
    o.y = h->logits; o.ld = c.vocab; o.write_logits = (logits_rows == n) ? want_logits : 1;
    o.ssq_in = h->ssq + (size_t)first * nt; o.nt_in = nt; o.hidden = H; o.eps = c.rms_eps;
    o.stats = h->stats; o.mask_id = c.mask_id;
    TcGroup lm = group(h->a, h->a_lo, (size_t)first * H, m, H, 1, table, c.vocab, nullptr, 0, nullptr, 0);
    set_rows(&lm, h->a, h->a_lo, (size_t)first * H, h->head_fmt);
    if (!c.tie_embeddings) lm.scale[0] = h->w.s_lm_head;
    if (!gemm(lm, o))
      return fail(h, FDVLM_ERR_CUDA, "lm head launch: %s", cudaGetErrorString(e));
    if (logits_rows == n) {
      launch_stats_merge(h->stats, ceil_div(c.vocab, 128) * 4, n, h->conf, h->pred, h->st, stamp(FDVLM_K_STATS_MERGE));
      h->launches++;
    }
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return fail(h, FDVLM_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(e));
  return FDVLM_OK;
}

// The kernels of one forward (with the ends of a step) on the handle's stream.  len_ptr: cache length from device memory.
static int enqueue_rows(fdvlm_t* h, int n, int mode, int logits_rows, int want_logits, const int* len_ptr, bool stamped, const StepEnds& ends,
                        bool sel_from_device) {
  int rc;
  if (ends.tokens) {
    rc = stage_rows(h, 0, n, ends.tokens, nullptr, mode, len_ptr);
    if (rc) return rc;
  }
  rc = h->use_tc ? forward_rows_tc(h, n, mode, logits_rows, want_logits, len_ptr, stamped)
                 : forward_rows_f32(h, n, mode, logits_rows, want_logits, len_ptr, ends.tokens != nullptr);
  if (rc || !ends.sel) return rc;
  const float* conf = h->conf + ends.sel_row0;
  const int32_t* pred = h->pred + ends.sel_row0;
  if (sel_from_device)
    launch_select_dev(conf, pred, h->blk_tokens, h->blk_masked, h->unmask, h->info, n - ends.sel_row0, h->dev_step, h->st);
  else
    launch_select(conf, pred, h->blk_tokens, h->blk_masked, h->unmask, h->info, n - ends.sel_row0, (int)ends.sel->rule, ends.sel->threshold,
                  ends.sel->k, h->st, ends.sel->pred_shift);
  h->launches++;
  CU(h, cudaGetLastError());
  return FDVLM_OK;
}

// The forward as a replayed CUDA graph: every kernel takes the cache length from a device word, so one capture per (rows,
// mode, logits mode, ends, stamped or not) serves every later call; the programmatic-dependent-launch edges are kept.
static int forward_rows_graph(fdvlm_t* h, int n, int mode, int logits_rows, int want_logits, const StepEnds& ends) {
  const int stamped = (h->prof_on == 2) ? 1 : 0, staged = ends.tokens ? 1 : 0, sel_row0 = ends.sel ? ends.sel_row0 : -1;
  set_dev_len(h);
  if (ends.sel) {
    const StepDev v = {(int)ends.sel->rule, ends.sel->threshold, ends.sel->k, ends.sel->pred_shift};
    const StepDev& w = h->step_set;
    if (v.rule != w.rule || v.threshold != w.threshold || v.k != w.k || v.shift != w.shift) {
      launch_set_step(h->dev_step, v, h->st);
      h->launches++;
      h->step_set = v;
    }
  }
  if (stamped) CU(h, cudaMemsetAsync(h->stamps, 0xFF, sizeof(KStamp) * FDVLM_MAX_STAMPS, h->st));
  for (auto& g : h->graphs) {
    if (g.n == n && g.mode == mode && g.logits_rows == logits_rows && g.want_logits == want_logits && g.stamped == stamped && g.staged == staged &&
        g.sel_row0 == sel_row0) {
      if (stamped) {      // the records' kinds are those of the capture: replay the bookkeeping only
        h->stamp_kind = g.kinds;
        h->stamp_used = (int)g.kinds.size();
      }
      CU(h, cudaGraphLaunch(g.exec, h->st));
      h->launches += g.launches;
      return FDVLM_OK;
    }
  }
  const int before = h->launches;
  CU(h, cudaStreamBeginCapture(h->st, cudaStreamCaptureModeThreadLocal));
  const int rc = enqueue_rows(h, n, mode, logits_rows, want_logits, h->dev_len, stamped != 0, ends, true);
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamEndCapture(h->st, &graph);
  if (rc != FDVLM_OK) { if (graph) cudaGraphDestroy(graph); return rc; }
  if (e != cudaSuccess) return fail(h, FDVLM_ERR_CUDA, "graph capture: %s", cudaGetErrorString(e));
  fdvlm::FwdGraph g;
  g.n = n; g.mode = mode; g.logits_rows = logits_rows; g.want_logits = want_logits; g.stamped = stamped; g.staged = staged; g.sel_row0 = sel_row0;
  g.launches = h->launches - before; g.exec = nullptr;
  if (stamped) g.kinds = h->stamp_kind;
  e = cudaGraphInstantiate(&g.exec, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) return fail(h, FDVLM_ERR_CUDA, "graph instantiate: %s", cudaGetErrorString(e));
  h->graphs.push_back(g);
  CU(h, cudaGraphLaunch(g.exec, h->st));
  return FDVLM_OK;
}

// The kernels of one tensor-core forward enqueued on the handle's stream, cache length taken from the device word:
// what a caller that is itself capturing the stream (the on-device decode loop) records.
int forward_rows_enqueue(fdvlm_t* h, int n, int mode, int logits_rows, int want_logits) {
  return forward_rows_tc(h, n, mode, logits_rows, want_logits, h->dev_len, false);
}

static bool being_captured(cudaStream_t st) {
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(st, &status) == cudaSuccess && status != cudaStreamCaptureStatusNone;
}

int forward_rows(fdvlm_t* h, int n, int mode, int logits_rows, int want_logits, const StepEnds& ends) {
  // Event timing around each kernel needs the kernels launched one by one.  So does a stream that the caller is capturing: it
  // takes no second capture, and the caller's graph may be replayed when the device's length word holds something else.
  if (h->use_graphs && h->prof_on != 1 && !being_captured(h->st)) return forward_rows_graph(h, n, mode, logits_rows, want_logits, ends);
  const bool stamped = h->prof_on == 2;
  if (stamped) CU(h, cudaMemsetAsync(h->stamps, 0xFF, sizeof(KStamp) * FDVLM_MAX_STAMPS, h->st));
  return enqueue_rows(h, n, mode, logits_rows, want_logits, nullptr, stamped, ends, false);
}

}  // namespace fdk
