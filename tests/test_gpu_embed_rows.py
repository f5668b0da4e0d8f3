"""The embedding step (token, position and type rows, LayerNorm or the next input's standardisation) at the row lengths where
its kernel changes shape, for few and many tokens, against the oracle through a prompt pass of a narrow two-layer model."""
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


@pytest.mark.parametrize("family,dtype", [(synth.GPT2, "bf16"), (synth.BERT, "bf16"), (synth.LLAMA, "f32")])
@pytest.mark.parametrize("D", [768, 776, 1024, 1032, 4104])
@pytest.mark.parametrize("P", [3, 21])
def test_embedding_row_lengths(family, dtype, D, P):
    cfg = synth.ModelConfig(family=family, n_layers=3, d_model=D, n_heads=2, head_dim=64, d_ffn=64, vocab=101, max_pos=64,
                            n_classes=3 if family == synth.BERT else 0, dtype=dtype, hsm_m1=64, hsm_m2=64, max_batch=1,
                            max_seq=32, max_pass_tokens=P)
    pair = Pair(cfg, seed=130)
    tokens = synth.make_tokens(131, 1, P, 101).numpy()
    compare_prefill(pair, tokens, 0.9, synth.forced_exits_uniform(132, P, 2, 3).numpy().reshape(1, P))
    pair.close()
