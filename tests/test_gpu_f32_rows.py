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
