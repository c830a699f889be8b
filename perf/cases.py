"""The work that a user of this library has it do, as cases that can be timed and compared.

A case is one request at batch size one: a prompt of vision-embedding rows and text tokens goes into the KV cache
(`prefill`), then an answer is decoded block by block (`answer`), or by one of the two self-speculative schemes (`spec`:
linear, Appendix B Alg. 1; `quad`: quadratic, Alg. 2).  The decoder shapes, prompt lengths, block sizes and rules are those
of `paper_2604_06832_b200.inputs.WORKLOADS`; `draw` spreads them over the ranges between.

Weights are N(0, 0.02) as everywhere in this repository, except that the first layer carries what a trained model has and
random weights lack: attention heads that look a fixed distance back (through the QKV biases, which Qwen2.5 has) and copy
the token found there into the residual stream.  So the model answers by copying from its prompt, with confidences spread
over (0, 1) and a clear winner at every position, and correct implementations decode the same tokens.
"""
from __future__ import annotations

import math

import torch

from paper_2604_06832_b200 import binding as B
from paper_2604_06832_b200 import inputs as I

# model: decoder shape, type of the KV cache (the 7B configuration prescribes bf16), strength of the copied token
# in the residual stream and gain of the last norm (which set how confident the model is)
MODELS = {
    "tiny": (I.TINY, B.KV_F16, 4.0, 1.0),
    "3b": (I.QWEN3B, B.KV_F16, 14.0, 1.2),
    "7b_fp8": (I.QWEN7B_FP8, B.KV_BF16, 9.0, 1.0),
    "7b_w8a8": (I.QWEN7B_FP8.with_(dtype=I.W8A8), B.KV_BF16, 9.0, 1.0),
}


def listed():
    # `prefix`: positions in the cache before the call; `rows`: prompt rows that the call appends (a quarter of each is
    # text tokens, the rest vision embeddings); `blocks`: blocks of `block` tokens decoded by the call; `k` > 0: top-k
    # rule, k = 0: confidence threshold 0.9; `host`: the caller steps the block itself and reads every step's results.
    return [
        # the smallest model in exact fp32, stepped from the host: launches and round trips are all that counts
        {"name": "answer_tiny_f32_host", "kind": "answer", "model": "tiny", "prefix": 64, "block": 8, "blocks": 1, "k": 0, "host": True},
        # the headline workload: 64 tokens of an answer behind an image and a question, 8 tokens a step
        {"name": "answer_3b_p1024_b32", "kind": "answer", "model": "3b", "prefix": 1024, "block": 32, "blocks": 2, "k": 8, "host": False},
        # several high-resolution images: the cache is as long as it gets
        {"name": "answer_3b_p8192_b32", "kind": "answer", "model": "3b", "prefix": 8192, "block": 32, "blocks": 1, "k": 8, "host": False},
        # the smallest block size of the sweep, threshold rule: few rows to a forward
        {"name": "answer_3b_p2048_b4", "kind": "answer", "model": "3b", "prefix": 2048, "block": 4, "blocks": 4, "k": 0, "host": False},
        # the largest block: 64 rows to a forward, each block committed by a pass of its own
        {"name": "answer_3b_p2048_b64", "kind": "answer", "model": "3b", "prefix": 2048, "block": 64, "blocks": 1, "k": 0, "host": False},
        # the larger model with FP8 weights, and with the projections' inputs quantised as well
        {"name": "answer_7b_fp8_p1024_b32", "kind": "answer", "model": "7b_fp8", "prefix": 1024, "block": 32, "blocks": 1, "k": 0, "host": False},
        {"name": "answer_7b_w8a8_p1024_b32", "kind": "answer", "model": "7b_w8a8", "prefix": 1024, "block": 32, "blocks": 1, "k": 0, "host": False},
        # the paper's self-speculative schemes
        {"name": "spec_3b_p2048_b32", "kind": "spec", "model": "3b", "prefix": 2048, "block": 32, "blocks": 2},
        {"name": "quad_3b_p1024_b5", "kind": "quad", "model": "3b", "prefix": 1024, "block": 5, "blocks": 4},
        # prompts: one image with a question, many images, a ragged one on the larger model
        {"name": "prefill_3b_1024", "kind": "prefill", "model": "3b", "prefix": 0, "rows": 1024},
        {"name": "prefill_3b_8192", "kind": "prefill", "model": "3b", "prefix": 0, "rows": 8192},
        {"name": "prefill_7b_fp8_1531", "kind": "prefill", "model": "7b_fp8", "prefix": 0, "rows": 1531},
    ]


def _spread(rng, lo, hi):
    """A whole number of [lo, hi], evenly over its logarithm."""
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(("answer", "answer", "answer", "prefill", "prefill", "spec", "quad"))
    model = rng.choice(("3b", "3b", "3b", "7b_fp8", "7b_fp8", "tiny", "7b_w8a8"))
    if kind == "prefill":
        # the first prompt, or a further turn behind what is already there (W8A8: see tolerance())
        model = "7b_fp8" if model == "7b_w8a8" else model
        rows = _spread(rng, 16, {"tiny": 1024, "3b": 8192, "7b_fp8": 2500}[model])
        prefix = 0 if rng.random() < 0.6 else _spread(rng, 64, 1024 if model == "tiny" else 8192 - min(rows, 8000))
        return {"kind": kind, "model": model, "prefix": prefix, "rows": rows}
    prefix = _spread(rng, 48, 1024) if model == "tiny" else _spread(rng, 700, 8192)
    if kind == "answer":
        host = model == "tiny" or rng.random() < 0.2
        block = _spread(rng, 2, 16) if model == "tiny" else _spread(rng, 2, 64)
        blocks = max(1, min(4, 64 // block))
        return {"kind": kind, "model": model, "prefix": prefix, "block": block, "blocks": rng.randint(1, blocks),
                "k": rng.choice((0, 0, 4, 8)), "host": host}
    if kind == "spec":
        return {"kind": kind, "model": model, "prefix": prefix, "block": _spread(rng, 2, 64), "blocks": rng.randint(1, 3)}
    return {"kind": kind, "model": model, "prefix": prefix, "block": rng.randint(2, 7), "blocks": rng.randint(2, 6)}


def _make_model(model, seed, reach):
    """The weights of `model`; its first layer copies the token `reach` positions back."""
    shape, _, strength, gain = MODELS[model]
    w = I.make_weights(shape, seed, qkv_bias=True, final_gain=gain, device="cuda")
    fp8 = shape.dtype in (I.FP8, I.W8A8)

    def values(lw, name):
        return lw[name].view(torch.float8_e4m3fn).float() * lw[I._SCALE_NAMES[name]][:, None] if fp8 else lw[name].float()

    def store(x):
        return I.quantize_e4m3_rows(x) if fp8 else (x.to(w["embed"].dtype), None)

    # the score of a key at distance D is sum_j u^2 cos((D - reach) theta_j) / sqrt(d) over the fast rotary frequencies
    lw, d = w["layers"][0], shape.head_dim
    j = torch.arange(d // 2, device="cuda", dtype=torch.float64)
    angle = reach * shape.rope_theta ** (-2.0 * j / d)
    u = torch.where(j < d // 4, 8.0, 0.0).double()
    lw["bq"] = torch.cat([u, torch.zeros_like(u)]).float().repeat(shape.n_q_heads)
    lw["bk"] = torch.cat([u * angle.cos(), u * angle.sin()]).float().repeat(shape.n_kv_heads)
    for name in ("wq", "wk"):                      # where the head looks does not depend on what is there
        lw[name], lw[I._SCALE_NAMES[name]] = store(0.1 * values(lw, name))
    group = shape.n_q_heads // shape.n_kv_heads
    v = values(lw, "wv").view(shape.n_kv_heads, 1, d, shape.hidden).expand(-1, group, -1, -1).reshape(shape.q_dim, shape.hidden)
    s = strength / (group * math.sqrt(shape.kv_dim * shape.hidden) * 0.02 * 0.02)
    lw["wo"], lw["s_o"] = store((s * v).t().contiguous())
    if not shape.tie_embeddings:                   # the head reads out what the embedding put in
        w["lm_head"], w["s_lm_head"] = store(w["embed"].float())
    return w


def _make_rows(shape, n, seed):
    """A prompt of n rows: three quarters vision embeddings ~ N(0, 1), the rest text tokens."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ne = n * 3 // 4
    emb = torch.randn(ne, shape.hidden, generator=gen, device="cuda").to(torch.float32 if shape.dtype == I.F32 else torch.bfloat16)
    tok = torch.randint(0, shape.vocab - 1, (n - ne,), generator=gen, device="cuda", dtype=torch.int32)
    return emb, tok + (tok >= shape.mask_id).to(torch.int32)


def prepare(case, seed):
    shape, kv, _, _ = MODELS[case["model"]]
    L, block, blocks, rows = case["prefix"], case.get("block", 0), case.get("blocks", 0), case.get("rows", 0)
    # (the answer copies text of the prompt: the last eighth to quarter of it)
    weights = _make_model(case["model"], seed, 3 * (L + rows) // 16)
    stream = torch.cuda.Stream()
    handle = B.Handle(shape, weights, max_seq=L + rows + blocks * block + 128, max_block=64, stream=stream, kv_dtype=kv)
    emb, tok = _make_rows(shape, L, 7 * seed + 1)
    first = torch.empty(shape.vocab, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    if L:
        handle.prefill(emb, tok, first)
        handle.synchronize()
    s = {"case": case, "handle": handle, "stream": stream,
         "logits": torch.zeros(shape.vocab, dtype=torch.float32, device="cuda")}
    ints = lambda *n: torch.zeros(n, dtype=torch.int32, device="cuda")
    if case["kind"] == "prefill":
        s["emb"], s["tok"] = _make_rows(shape, rows, 7 * seed + 2)
    elif case["kind"] == "answer" and case["host"]:
        s["tokens"] = torch.zeros(blocks, block, dtype=torch.int32).pin_memory()
        s["conf"] = torch.zeros(block, dtype=torch.float32).pin_memory()
        s["pred"] = torch.zeros(block, dtype=torch.int32).pin_memory()
    elif case["kind"] == "answer":
        s["tokens"] = ints(blocks, block)
    else:
        first[shape.mask_id] = -math.inf
        s["first"] = int(first.argmax())           # the token that the prompt's last row predicts
        s["draft"], s["verify"] = ints(blocks, block), ints(blocks, block)
        s["rows"] = ints(blocks, block * (block + 1))
    torch.cuda.synchronize()
    return s


def run(s):
    case, h = s["case"], s["handle"]
    block, blocks = case.get("block", 0), case.get("blocks", 0)
    h.truncate(case["prefix"])                     # back to the conversation as it stood before this turn
    if case["kind"] == "prefill":
        h.prefill(s["emb"], s["tok"], s["logits"])
        # every position's K and V of the last layer: what all layers made of the prompt
        with torch.cuda.stream(s["stream"]):
            kv = [h.cache_read(h.shape.n_layers - 1, which, case["prefix"], case["rows"]) for which in (0, 1)]
        return {"logits": s["logits"], "k": kv[0], "v": kv[1]}
    if case["kind"] == "spec":
        seed, accepted = s["first"], []
        for i in range(blocks):
            info = h.spec_block(block, seed, s["draft"][i], s["verify"][i])
            seed = info.next_token
            accepted.append(info.accepted)
        return {"draft": s["draft"], "verify": s["verify"], "accepted": accepted, "next": seed}
    if case["kind"] == "quad":
        h.quad_begin(block, s["first"])
        accepted = [h.quad_step(s["verify"][i], s["draft"][i], s["rows"][i]).accepted for i in range(blocks)]
        h.quad_end()
        return {"tokens": s["verify"], "draft": s["draft"], "rows": s["rows"], "accepted": accepted}
    rule = B.RULE_TOPK if case["k"] else B.RULE_THRESHOLD
    joined = 2 * block <= 64                       # a block's commit can ride in the next block's first forward
    for i in range(blocks):
        if case["host"]:
            h.block_begin_host(block)
            while h.block_step_host(rule, 0.9, case["k"], conf=s["conf"], pred=s["pred"], block_tokens=s["tokens"][i]).n_remaining:
                pass
        elif case["k"]:
            (h.commit_decode_block_topk if joined else h.decode_block_topk)(block, case["k"], block_tokens=s["tokens"][i])
        else:
            (h.commit_decode_block if joined else h.decode_block)(block, rule, 0.9, block_tokens=s["tokens"][i])
        if case["host"] or not joined or i + 1 == blocks:
            h.commit_block(s["logits"])
    # W8A8: the tokens alone, see tolerance()
    return {"tokens": s["tokens"]} if case["model"] == "7b_w8a8" else {"tokens": s["tokens"], "logits": s["logits"]}


def work(case):
    """Every weight and every cached position once for each forward that the schedule cannot do without, and two operations
    for each weight and row.  The threshold rule's forwards depend on the confidences: one is the least there can be."""
    shape = MODELS[case["model"]][0]
    L, layer_weights = case["prefix"], shape.linear_elements() - shape.vocab * shape.hidden
    attention = lambda n, keys: 4 * shape.n_layers * shape.q_dim * n * keys
    kv = shape.kv_bytes_per_token()
    if case["kind"] == "prefill":
        n = case["rows"]
        return {"bytes": shape.weight_bytes() + kv * (L + n) + n * shape.hidden * 2,
                "flops": 2 * layer_weights * n + attention(n, L + n / 2) + 2 * shape.vocab * shape.hidden}
    block, blocks = case["block"], case["blocks"]
    if case["kind"] == "quad":
        n, forwards = block * (block + 1), blocks
    elif case["kind"] == "spec":
        n, forwards = block, 2 * blocks
    else:
        n, forwards = block, blocks * (-(-block // case["k"]) if case["k"] else 1) + 1
    return {"bytes": forwards * (shape.weight_bytes() + kv * L),
            "flops": forwards * (2 * shape.linear_elements() * n + attention(n, L + n))}


def tolerance(case):
    # Tokens are the same: the model's winners are clear.  Logits and cached K / V pass through 16-bit q, K, V and GEMM
    # inputs in every layer.  A W8A8 forward rounds its inputs to 4 significant bits, where the last bit of a sum decides
    # between two codes: after a few layers two correct implementations differ by as much as the quantisation itself, so of
    # those cases the tokens are compared and nothing else.
    return {"rel": 1e-5, "max": 1e-4} if case["model"] == "tiny" else {"rel": 1e-2, "max": 0.15}
