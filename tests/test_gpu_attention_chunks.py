"""Generation-step attention whose grid covers more chunks than a token has keys: contexts of one chunk, at a chunk's edge and
growing over it, capacities of one to many chunks, grouped and single heads, sequences that leave at different layers, against
the oracle."""
import numpy as np
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


@pytest.mark.parametrize("heads,kv,dh", [(4, 1, 128), (4, 2, 64), (2, 2, 64), (2, 2, 128)])
@pytest.mark.parametrize("P,max_seq", [(5, 1000), (126, 250), (255, 600)])
def test_chunks_past_the_context(heads, kv, dh, P, max_seq):
    cfg = synth.ModelConfig(family=synth.LLAMA, n_layers=4, d_model=256, n_heads=heads, n_kv_heads=kv, head_dim=dh, d_ffn=256,
                            vocab=500, dtype="bf16", hsm_m1=128, hsm_m2=256, max_batch=3, max_seq=max_seq,
                            max_pass_tokens=3 * P, block_shuffle_seed=7)
    pair = Pair(cfg, seed=150)
    ores, cache, _ = compare_prefill(pair, synth.make_tokens(151, 3, P, 500).numpy(), 2.0)
    compare_decode(pair, cache, ores.next_token, 4, 0.9, np.array([[4, 2, 3], [2, 4, 4], [3, 3, 2], [4, 4, 4]]))
    pair.compare_cache(cache, 3, P + 4)
    pair.close()
