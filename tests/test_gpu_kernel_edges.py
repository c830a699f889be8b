"""GPU parity where a kernel's split of the work changes: the branches that the small models of the other files do not reach."""
import numpy as np
import pytest
import torch

from oracle import fdvlm_oracle as orc
from paper_2604_06832_b200 import inputs as I

from helpers import make_pair, replay_decode, upload_prefix
from test_gpu_prefill import BF16, FP8, check

pytestmark = pytest.mark.gpu


# ---- decode attention: one warp per (row, head) in the merge, more chunks than it takes at a time, chunks longer than the ring ----
@pytest.mark.parametrize("elem", [torch.bfloat16, torch.float16], ids=["bf16", "f16"])
@pytest.mark.parametrize("n,L,hq,hkv,d,causal", [(64, 3000, 16, 2, 128, 0), (64, 9000, 16, 2, 128, 1), (64, 4100, 32, 8, 64, 1),
                                                 (8, 18000, 8, 1, 128, 0), (37, 2500, 28, 4, 128, 1)])
def test_decode_attention_chunks_and_merge(elem, n, L, hq, hkv, d, causal):
    from paper_2604_06832_b200 import binding as B
    g = torch.Generator().manual_seed(n + L)
    q, kc, vc = (torch.randn(*s, generator=g).to(elem) for s in ((n, hq, d), (hkv, L + n + 5, d), (hkv, L + n + 5, d)))
    T = L + n
    allowed = np.ones((n, T), dtype=bool)
    if causal:
        allowed[:, L:] = np.tril(np.ones((n, n), dtype=bool))
    f = lambda t: t.double().numpy()
    ref = orc.attend(f(q), f(kc)[:, :T].transpose(1, 0, 2), f(vc)[:, :T].transpose(1, 0, 2), allowed).reshape(n, hq * d)
    out = B.op_attention(q.cuda(), kc.cuda(), vc.cuda(), L, bool(causal), dtype=B.DT_BF16)
    torch.cuda.synchronize()
    # P is rounded to the element type (relative 2^-9 or 2^-12): a sum of p v with sum p = 1 moves by at most that times max |v|,
    # and the result is rounded once more
    eps = 2.0 ** -9 if elem == torch.bfloat16 else 2.0 ** -12
    bound = 2 * eps * float(vc.float().abs().max())
    assert np.abs(out.double().cpu().numpy() - ref).max() <= bound


# ---- callers' tensors need no more alignment than their elements where the loads and stores are no bulk copies ----
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("elem", [torch.float32, torch.bfloat16, torch.float16], ids=["f32", "bf16", "f16"])
def test_attention_operator_on_tensors_at_any_element(elem, d):
    from paper_2604_06832_b200 import binding as B
    n, L, hq, hkv, seq = 5, 70, 4, 2, 80
    g = torch.Generator().manual_seed(d)
    q, kc, vc = (torch.randn(*s, generator=g).to(elem).cuda() for s in ((n, hq, d), (hkv, seq, d), (hkv, seq, d)))
    f32 = elem == torch.float32
    dt, kv = (B.DT_F32 if f32 else B.DT_BF16), (B.KV_BF16 if elem == torch.bfloat16 else B.KV_F16)
    want = B.op_attention(q, kc, vc, L, True, dtype=dt)
    ws = torch.zeros(B.lib().fdvlm_op_attention_workspace_bytes(n, hq, hkv, d), dtype=torch.uint8, device="cuda")
    for off in (1, 2, 3):
        out = torch.zeros(want.numel() + 4, dtype=elem, device="cuda")
        args = [q, kc, vc]
        if f32:       # (the 16-bit kernels fetch these with 16-byte copies)
            args = [torch.zeros(t.numel() + 4, device="cuda")[off:off + t.numel()].copy_(t.flatten()) for t in args]
        rc = B.lib().fdvlm_op_attention(*(t.data_ptr() for t in args), out[off:].data_ptr(), n, L, seq, hq, hkv, d, 1, dt, kv, ws.data_ptr(), None)
        assert rc == 0
        torch.cuda.synchronize()
        assert torch.equal(out[off:off + want.numel()], want.flatten()) and not out[:off].any() and not out[off + want.numel():].any()


@pytest.mark.parametrize("shape", [I.TINY, BF16, FP8], ids=["f32", "bf16", "fp8"])
def test_norm_gains_at_any_element(shape):
    from paper_2604_06832_b200 import binding as B
    w = B.weights_to_device(I.make_weights(shape, 3, gain_spread=0.5))
    toks = I.random_tokens(shape, 150, 4).cuda()
    outs = []
    for off in (0, 1):
        for t in [w] + w["layers"]:
            for name in ("g_final", "g_attn", "g_mlp"):
                if name in t:
                    t[name] = torch.zeros(shape.hidden + 4, device="cuda")[off:off + shape.hidden].copy_(t[name])
        h = B.Handle(shape, w, max_seq=256)
        last = torch.empty(shape.vocab, device="cuda")
        h.prefill(None, toks, last)
        h.synchronize()
        outs.append(last)
        h.close()
    assert torch.equal(*outs)


# ---- SwiGLU of gates outside the range of its arithmetic ----
@pytest.mark.parametrize("n", [5, 150], ids=["decode", "prompt"])
def test_an_infinite_gate_saturates_like_a_large_one(n):
    """A gate of +inf gives an activation that is stored as +-65504, as one of 1e7 does.  (fp8 weights, whose activations are f16 values;
    all entries of the embedding rows are positive and dominate the residual stream, so the gate of the feature is.)"""
    from paper_2604_06832_b200 import binding as B
    shape = FP8.with_(n_layers=1)
    w = B.weights_to_device(I.make_weights(shape, 3))
    lw, feature = w["layers"][0], 37
    lw["w_gate"][feature] = 0x38                                  # e4m3 code of 1.0
    lw["w_up"][feature] = 0x38                                    # (far above 65504 / 1e7 too)
    emb = torch.ones(n, shape.hidden, dtype=torch.bfloat16, device="cuda")
    outs = []
    for scale in (1e7 / shape.hidden, 3e38):
        lw["s_gate"][feature] = scale
        h = B.Handle(shape, w, max_seq=256)
        last = torch.empty(shape.vocab, device="cuda")
        h.prefill(emb, None, last)
        h.synchronize()
        outs.append(last)
        h.close()
    assert torch.isfinite(outs[0]).all() and torch.equal(*outs)


# ---- exact fp32: a NaN logit spoils the confidences and is never the prediction ----
@pytest.mark.parametrize("step", [8, -8, 1], ids=["same-pair-above", "same-pair-below", "next-pair"])
def test_exact_f32_prediction_beside_a_nan_logit(step):
    from paper_2604_06832_b200 import binding as B
    w = B.weights_to_device(I.make_weights(I.TINY, 6))
    toks = torch.arange(40, dtype=torch.int32, device="cuda")
    pred, conf = torch.empty(1, dtype=torch.int32, device="cuda"), torch.empty(1, device="cuda")

    def predict():
        h = B.Handle(I.TINY, w, max_seq=64)
        h.prefill(None, toks)
        h.block_begin(1)
        h.block_step(B.RULE_TOPK, 0.0, 1, pred=pred, conf=conf)
        h.close()
        return int(pred), float(conf)

    target = 304 + (8 if step == -8 else 0)                       # lane 0 of a tile of 16 ids, as its lower or upper one
    mask_row = w["embed"][I.TINY.mask_id].clone()
    for gain in (1.0, 4.0, 16.0, 64.0):                           # until the id wins: its row points along the mask row
        w["embed"][target] = gain * mask_row
        best, c = predict()
        if best == target:
            break
    assert best == target and np.isfinite(c)
    w["embed"][target + step] = float("nan")
    best, c = predict()
    assert best == target and np.isnan(c)


# ---- exact fp32: depth beyond one shared-memory panel, ragged widths, every row tile, more keys than one pass holds ----
WIDE_F32 = I.TINY.with_(n_layers=1, hidden=1096, intermediate=1112, vocab=1003, mask_id=1002)


@pytest.mark.parametrize("n", [1, 7, 9, 17, 33])
def test_exact_f32_row_tiles_and_ragged_widths(n):
    check(WIDE_F32, [(0, n)])


@pytest.mark.parametrize("n", [33, 64])
def test_exact_f32_wide_layers(n):
    """Widths from which 32 rows take two pairs of features a lane, the last tile of each ragged: every projection, and the statistics."""
    shape = I.TINY.with_(n_layers=1, hidden=2376, n_q_heads=32, n_kv_heads=4, intermediate=1192, vocab=2399, mask_id=1200)
    oracle, handle, _ = make_pair(shape, 5, max_seq=128, qkv_bias=True)
    emb, toks = I.make_prefix(shape, 20, 20, 3)
    oracle.prefill(I.as_numpy_storage(emb), toks.numpy())
    handle.prefill(*upload_prefix(emb, toks))
    stats = replay_decode(oracle, handle, shape, n, orc.TOPK, 0.0, n)
    assert stats["steps"] == 1 and stats["rows_sure"] > 0
    handle.close()


def test_exact_f32_attention_over_many_keys():
    check(I.TINY.with_(n_layers=1), [(0, 2100), (0, 9)], max_seq=2200)


# ---- prompts: tiles of the last wave in pieces along k, 256-row attention CTAs ----
@pytest.mark.parametrize("shape,n", [
    (BF16.with_(n_layers=1, hidden=1536, intermediate=2560, vocab=512, mask_id=511), 770),                        # gate/up
    (BF16.with_(n_layers=1, hidden=2048, n_q_heads=16, intermediate=1536, vocab=512, mask_id=511), 2310),         # QKV, O, down
    (FP8.with_(n_layers=1, hidden=2048, n_q_heads=32, n_kv_heads=4, intermediate=1792, vocab=512, mask_id=511), 1290)],
    ids=["bf16-gate-up", "bf16-qkv-o-down", "fp8-gate-up"])
def test_prompt_tiles_in_pieces(shape, n):
    check(shape, [(n - 100, 100)])


# ---- the captured step: rule and threshold change between replays of one graph ----
@pytest.mark.parametrize("shape", [I.TINY, BF16], ids=["f32", "bf16"])
def test_captured_step_follows_its_parameters(shape):
    stream = torch.cuda.Stream()
    oracle, handle, _ = make_pair(shape, 5, max_seq=128, stream=stream)
    emb, toks = I.make_prefix(shape, 30, 10, 3)
    oracle.prefill(I.as_numpy_storage(emb), toks.numpy())
    with torch.cuda.stream(stream):       # (the commit is only enqueued: its logits are read back on the handle's own stream)
        handle.prefill(*upload_prefix(emb, toks))
        for rule, tau, k in ((orc.THRESHOLD, 0.9, 0), (orc.TOPK, 0.0, 3), (orc.TOPK, 0.0, 5), (orc.THRESHOLD, 1e-4, 0)):
            replay_decode(oracle, handle, shape, 8, rule, tau, k)
        handle.synchronize()
    handle.close()


# ---- fp8 weights: the byte planes of rows whose values span the range of f16 ----
def test_fp8_projection_of_rows_with_small_values():
    from paper_2604_06832_b200 import binding as B
    g = torch.Generator().manual_seed(3)
    m, n, k = 40, 300, 640
    x = (torch.randn(m, k, generator=g) * 10.0 ** (-7.0 * torch.rand(m, k, generator=g))).to(torch.bfloat16)
    codes, scale = I.quantize_e4m3_rows(torch.randn(n, k, generator=g) * 0.02)
    w = orc.to_f64(codes.numpy()) * scale.double().numpy()[:, None]
    xv = x.double().numpy()
    y = B.op_linear(x.cuda(), codes.cuda(), scale.cuda(), None, dtype=B.DT_FP8).double().cpu().numpy()
    # f16 of a bf16 value and its planes are exact from 2^-13 up and off by at most 2^-24 below; fp32 sums of k products
    bound = (2.0 ** -24 + 2.0 ** -25) * np.abs(w).sum(1)[None] + 2.0 ** -20 * (np.abs(xv) @ np.abs(w).T)
    assert (np.abs(y - xv @ w.T) <= bound).all()


# ---- gate / up of a decode step, one share of the features per SM: row counts at which the planes change, ragged last share and depth ----
@pytest.mark.parametrize("base,inter,n", [(BF16, 2384, 1), (BF16, 2384, 16), (BF16, 2384, 17), (BF16, 2384, 33), (BF16, 2384, 64), (BF16, 1216, 31), (BF16, 19008, 24),
                                          (FP8, 2416, 3), (FP8, 4816, 3), (FP8, 2416, 33), (FP8, 2416, 40), (FP8, 2416, 41), (FP8, 2416, 49), (FP8, 2416, 64)])
def test_gate_up_shares(base, inter, n):
    """(19008 features are more than 128 per SM and stay with the tiles, as do 2416 of fp8 weights up to 8 rows; hidden: a last tile of 80 columns in the finalisation.)"""
    shape = base.with_(n_layers=1, hidden=1104, intermediate=inter)
    oracle, handle, _ = make_pair(shape, 5, max_seq=128, qkv_bias=True)
    emb, toks = I.make_prefix(shape, 20, 20, 3)
    oracle.prefill(I.as_numpy_storage(emb), toks.numpy())
    handle.prefill(*upload_prefix(emb, toks))
    assert replay_decode(oracle, handle, shape, n, orc.TOPK, 0.0, n)["steps"] == 1
    handle.close()


@pytest.mark.parametrize("shape,n", [(BF16, 33), (FP8, 64)], ids=["bf16", "fp8"])
def test_give_up_path_of_the_gate_up_shares(shape, n):
    """With the poison flag set every role leaves as after a wait that timed out; afterwards the step is what it was before, bit for bit."""
    from paper_2604_06832_b200 import binding as B
    h = B.Handle(shape, B.weights_to_device(I.make_weights(shape, 3)), max_seq=256, stream=torch.cuda.Stream())
    toks = I.random_tokens(shape, 40, 4).cuda()

    def step():
        logits = torch.empty(n, shape.vocab, device="cuda")
        h.reset()
        h.prefill(None, toks)
        h.block_begin(n)
        h.block_step(B.RULE_TOPK, 0.0, n, logits=logits)
        return logits

    before = step()
    h.debug_poison(True)
    with pytest.raises(B.FdvlmError) as e:
        step()
    assert e.value.code == B.ERR_TIMEOUT
    h.debug_poison(False)
    assert torch.equal(before, step())
    h.close()


@pytest.mark.parametrize("shape,n", [(BF16, 33), (BF16.with_(hidden=1104), 64), (FP8, 40), (FP8.with_(hidden=1104), 64), (FP8.with_(dtype=I.W8A8), 17),
                                     (BF16.with_(hidden=2048, intermediate=4096), 32), (FP8.with_(hidden=2048, intermediate=8192), 16)],
                         ids=["bf16", "bf16-deep", "fp8", "fp8-deep", "w8a8", "bf16-items", "fp8-items"])
def test_producers_that_do_not_hear_of_an_abort(shape, n):
    """The other roles give up before the producers issue anything.  Where all k-blocks fit into the ring no wait of a producer fails, and
    the CTA must wait for its copies all the same; afterwards the step is what it was before, bit for bit."""
    from paper_2604_06832_b200 import binding as B
    h = B.Handle(shape, B.weights_to_device(I.make_weights(shape, 3)), max_seq=256, stream=torch.cuda.Stream())
    toks = I.random_tokens(shape, 40, 4).cuda()

    def step():
        logits = torch.empty(n, shape.vocab, device="cuda")
        h.reset()
        h.prefill(None, toks)
        h.block_begin(n)
        h.block_step(B.RULE_TOPK, 0.0, n, logits=logits)
        return logits

    before = step()
    for _ in range(2):
        h.debug_poison(2)
        with pytest.raises(B.FdvlmError) as e:
            step()
        assert e.value.code == B.ERR_TIMEOUT
        h.debug_poison(False)
        assert torch.equal(before, step())
    h.close()
