"""GPU parity of prompts: last-row logits and every layer's cached K / V against the oracle.  Prompts of up to 128 rows, and short ones
behind long caches, run through the decode path in forwards of max_block rows; all others through the prompt path (large-M GEMMs and
causal attention of whole row blocks), here at the edges of its tiles."""
import numpy as np
import pytest
import torch

from paper_2604_06832_b200 import inputs as I

from helpers import TOL, make_pair, upload_prefix

pytestmark = pytest.mark.gpu

BF16 = I.ModelShape(n_layers=2, hidden=512, n_q_heads=8, n_kv_heads=2, head_dim=128, intermediate=1376, vocab=4096, mask_id=4095,
                    tie_embeddings=True, dtype=I.BF16)
# widths that are no multiple of a tile; head_dim 64; an FP8 model with a tied bf16 head
RAGGED = BF16.with_(hidden=400, n_q_heads=6, n_kv_heads=3, head_dim=64, intermediate=912)
FP8 = BF16.with_(dtype=I.FP8, tie_embeddings=False, n_q_heads=4, n_kv_heads=4, head_dim=64, hidden=384, intermediate=1120, vocab=3000,
                 mask_id=2999)
FP8_TIED = BF16.with_(dtype=I.FP8)


def check(shape, parts, seed=5, max_seq=None, prompt_path=None, **kw):
    """Prompt given in `parts` = [(embedding rows, tokens), ...], one call each; prompt_path: which of them must take that path."""
    tol = TOL[shape.dtype]["logits"]      # K and V are projections of unit-rms rows like the logits: the same bound
    total = sum(a + b for a, b in parts)
    oracle, handle, _ = make_pair(shape, seed, max_seq=max_seq or total + 64, qkv_bias=True, **kw)
    last = torch.empty(shape.vocab, dtype=torch.float32, device="cuda")
    for i, (ne, nt) in enumerate(parts):
        emb, toks = I.make_prefix(shape, ne, nt, 10 + i)
        ref = oracle.prefill(I.as_numpy_storage(emb) if ne else None, toks.numpy() if nt else None)
        handle.prefill(*upload_prefix(emb, toks), last)
        handle.synchronize()
        assert handle.cache_len() == oracle.cache_len
        if prompt_path:      # (one forward of at most 8 launches a layer against a forward for every 64 rows)
            forwards = -(-(ne + nt) // 4096) if prompt_path[i] else -(-(ne + nt) // 64)
            per_forward = handle.last_launch_count() / forwards
            assert (per_forward <= 8 * shape.n_layers + 6) if prompt_path[i] else (per_forward >= 9 * shape.n_layers)
        assert np.abs(last.double().cpu().numpy() - ref).max() <= tol
    for l in range(shape.n_layers):
        for which, want in ((0, oracle.K[l]), (1, oracle.V[l])):
            got = handle.cache_read(l, which, 0, total)
            torch.cuda.synchronize()
            assert np.abs(got.double().cpu().numpy() - want).max() <= tol, (l, which)
    handle.close()


@pytest.mark.parametrize("n", [65, 127, 128, 129, 256, 257, 391])
@pytest.mark.parametrize("shape", [BF16, RAGGED, FP8, FP8_TIED], ids=["bf16", "ragged", "fp8", "fp8-tied"])
def test_prompt_at_the_edges_of_its_row_tiles(shape, n):
    check(shape, [(n * 3 // 4, n - n * 3 // 4)])


@pytest.mark.parametrize("shape", [BF16, FP8], ids=["bf16", "fp8"])
@pytest.mark.parametrize("parts", [[(0, 70), (0, 130)], [(100, 0), (3, 4), (0, 77)]], ids=["70+130", "100+7+77"])
def test_further_turn_behind_a_cached_prompt(shape, parts):
    check(shape, parts, stream=torch.cuda.Stream())


@pytest.mark.parametrize("kv", ["KV_F16", "KV_BF16"])
@pytest.mark.parametrize("shape", [BF16, RAGGED, FP8], ids=["bf16", "ragged", "fp8"])
def test_further_turns_of_the_prompt_path(shape, kv):
    """Each turn above 128 rows, behind caches whose lengths are no multiple of a tile (one of them more than 2000 positions)."""
    from paper_2604_06832_b200 import binding as B
    check(shape.with_(n_layers=1, vocab=512, mask_id=511), [(0, 201), (100, 231), (0, 1700), (130, 163)],
          stream=torch.cuda.Stream(), kv_dtype=getattr(B, kv), prompt_path=[True] * 4)


@pytest.mark.parametrize("before,prompt_path", [(5245, True), (5248, False)])
def test_short_turn_at_the_line_between_the_paths(before, prompt_path):
    """The rule weighs the keys against the forwards of the decode path: 150 rows of this shape cross at 5396 keys."""
    shape = BF16.with_(n_layers=1, hidden=256, n_q_heads=2, n_kv_heads=1, intermediate=512, vocab=512, mask_id=511)
    check(shape, [(0, before), (0, 150)], prompt_path=[True, prompt_path])


def test_prompt_of_several_forwards():
    """More rows than one forward takes: equal parts, each causal behind the ones before."""
    shape = BF16.with_(n_layers=1, hidden=256, n_q_heads=2, n_kv_heads=1, intermediate=512, vocab=512, mask_id=511)
    check(shape, [(0, 4300)])
