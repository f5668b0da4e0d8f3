"""How the tcgen05 prompt attention deals its work out: several heads of 64 per CTA when (tile, head) pairs exceed the SMs, the
sequences of a tile over several CTAs when they are few, against the oracle, with tokens leaving at every layer (so that both
change from layer to layer), tiles that end inside a sequence, and cross-attention over short prompts."""
import pytest
import torch

import synth
from parity_utils import Pair, compare_prefill

import paper_2601_03700_gb300 as adept

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    adept.load_library()


def config(family, B, P, heads, dh=64):
    return synth.ModelConfig(family=family, n_layers=4, d_model=heads * dh, n_heads=heads, head_dim=dh, d_ffn=512, vocab=777,
                             max_pos=256, n_classes=3 if family == synth.BERT else 0, dtype="bf16", hsm_m1=256, hsm_m2=512,
                             max_batch=B, max_seq=max(P + 4, 16), max_pass_tokens=B * P, block_shuffle_seed=6)


@pytest.mark.parametrize("family,B,P,heads,dh", [
    (synth.BERT, 20, 128, 12, 64),    # 240 pairs: 2 heads per CTA, then fewer tiles
    (synth.GPT2, 5, 200, 24, 64),     # causal, tiles that span two sequences, 8 tiles x 24 heads
    (synth.BERT, 33, 5, 4, 64),       # 2 tiles of 26 sequences each
    (synth.GPT2, 40, 7, 3, 64),
    (synth.LLAMA, 19, 9, 4, 128),
])
def test_attention_work_split_matches_oracle(family, B, P, heads, dh):
    pair = Pair(config(family, B, P, heads, dh), seed=120 + P)
    tokens = synth.make_tokens(121, B, P, 777).numpy()
    forced = synth.forced_exits_uniform(122 + P, B * P, 2, 4).numpy().reshape(B, P)
    compare_prefill(pair, tokens, 0.9, forced)
    pair.close()
