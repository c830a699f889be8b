"""GPU parity of the prompt path (prompts above 64 rows: large-M GEMMs and causal attention of whole row blocks) at the
edges of its tiles: last-row logits and every layer's cached K / V against the oracle."""
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


def check(shape, parts, seed=5, max_seq=None, **kw):
    """Prompt given in `parts` = [(embedding rows, tokens), ...], one call each."""
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


def test_prompt_of_several_forwards():
    """More rows than one forward takes: equal parts, each causal behind the ones before."""
    shape = BF16.with_(n_layers=1, hidden=256, n_q_heads=2, n_kv_heads=1, intermediate=512, vocab=512, mask_id=511)
    check(shape, [(0, 4300)])
