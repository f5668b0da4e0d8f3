"""Reading K/V out of the paged cache: whole and partial ranges, block edges, buffers at a 16-byte boundary and not,
both types and the three head sizes, equal to what a one-position read gives."""
import pytest
import torch

import synth
import paper_2601_03700_gb300 as adept

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    adept.load_library()


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("head_dim,kv_heads", [(32, 3), (64, 2), (128, 1)])
def test_ranges_and_alignments(dtype, head_dim, kv_heads):
    cfg = synth.ModelConfig(family=synth.LLAMA, n_layers=3, d_model=64, n_heads=kv_heads, head_dim=head_dim, d_ffn=64,
                            vocab=64, dtype=dtype, hsm_m1=64, hsm_m2=64, max_batch=2, max_seq=60, block_shuffle_seed=9)
    m = adept.Model(cfg, synth.make_weights(cfg, seed=4, std=0.1))
    m.prefill(synth.make_tokens(5, 2, 53, 64).cuda(), 9.0)
    per = kv_heads * head_dim
    one = [m.read_kv(2, 1, p, 1) for p in range(53)]
    want = [torch.cat([o[i] for o in one]).reshape(-1) for i in (0, 1)]
    assert want[0].float().norm() > 0 and not torch.equal(want[0], want[1])
    for p0, n in ((0, 53), (5, 30), (15, 2), (52, 1), (16, 16)):
        for shift in (0, 1, 8):
            buf = [torch.full((53 * per + 8,), -1.0, dtype=cfg.torch_dtype, device="cuda") for _ in range(2)]
            out = [b[shift:shift + n * per] for b in buf]
            adept.adept_read_kv(m.h, 2, 1, p0, n, *out)
            for o, w, b in zip(out, want, buf):
                assert torch.equal(o, w[p0 * per:(p0 + n) * per])
                assert (b[:shift] == -1).all() and (b[shift + n * per:] == -1).all()
    m.close()
