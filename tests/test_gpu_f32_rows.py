"""The fp32 GEMM of few rows (f32_rows_kernel) against the oracle: K below, at and above its 512-element slices over one,
two and four warps, outputs that are no multiple of its feature tiles (a ragged vocabulary among them), row counts
around its 8-row blocks and its bound, every epilogue (rotary, SwiGLU, GELU, residual, cache), both head sizes."""
import pytest
import torch

import synth
from parity_utils import Pair, compare_decode, compare_prefill

import paper_2601_03700_gb300 as adept

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    adept.load_library()


@pytest.mark.parametrize("family,head_dim", [(synth.LLAMA, 64), (synth.LLAMA, 128), (synth.GPT2, 64), (synth.BERT, 64)])
@pytest.mark.parametrize("B,P", [(1, 1), (1, 7), (4, 2), (3, 3), (1, 128), (3, 43), (2, 128)])
def test_f32_rows_match_oracle(family, head_dim, B, P):
    cfg = synth.ModelConfig(family=family, n_layers=4, d_model=264, n_heads=4, n_kv_heads=2, head_dim=head_dim,
                            d_ffn=1040, vocab=1003, max_pos=256, n_classes=3 if family == synth.BERT else 0,
                            dtype="f32", hsm_m1=520, hsm_m2=2056, max_batch=B, max_seq=P + 4,
                            max_pass_tokens=B * P, block_shuffle_seed=3)
    pair = Pair(cfg, seed=110 + P, std=0.04)
    tokens = synth.make_tokens(111, B, P, 1003).numpy()
    forced = synth.forced_exits_uniform(112 + P, B * P, 2, 4).numpy().reshape(B, P)
    ores, cache, _ = compare_prefill(pair, tokens, 0.9, forced)
    if family != synth.BERT:
        steps = synth.forced_exits_uniform(113, 3 * B, 2, 4).numpy().reshape(3, B)
        compare_decode(pair, cache, ores.next_token, 3, 0.9, steps)
        pair.compare_cache(cache, B, P + 3)
    pair.close()


@pytest.mark.parametrize("family,P", [(synth.LLAMA, 110), (synth.LLAMA, 111), (synth.LLAMA, 139), (synth.LLAMA, 250),
                                      (synth.GPT2, 250)])
def test_live_counts_on_both_sides_of_the_rule(family, P):
    """Wide products (16384 outputs of K 520: the rows kernel up to 110 rows and from 129 to 138, the tiles at the other
    counts; 8192 of the mapper up to 220), with live counts that fall from layer to layer across the line."""
    cfg = synth.ModelConfig(family=family, n_layers=6, d_model=520, n_heads=4, head_dim=64,
                            d_ffn=8192 if family == synth.LLAMA else 16384, vocab=517, max_pos=256, dtype="f32",
                            hsm_m1=520, hsm_m2=8192, max_batch=1, max_seq=P, max_pass_tokens=P, block_shuffle_seed=3)
    pair = Pair(cfg, weights=synth.make_weights(cfg, seed=130, std=0.03, device="cuda"))
    tokens = synth.make_tokens(131, 1, P, 517).numpy()
    compare_prefill(pair, tokens, 0.9, synth.forced_exits_uniform(132 + P, P, 2, 6).numpy().reshape(1, P))
    compare_prefill(pair, tokens, -2.0)      # every token leaves at layer 2: all rows to the mapper, none after it
    pair.close()
