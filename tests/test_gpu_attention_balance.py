"""bf16 prompts with heads of 32 (the attention without tensor cores) behind the paired GEMM: the attention's CTAs spread
over every SM.  Against the same launches without early starts, each timed alone, the pass is not slower: beside the
GEMM's last CTAs they crowded a third of the SMs, and the pass took 1.3 times as long (1.78 against 1.36 ms)."""
import pytest
import torch

import synth

import paper_2601_03700_gb300 as adept

pytestmark = pytest.mark.gpu


def test_prompt_behind_paired_gemm_is_not_slower_than_its_launches():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P = 512
    cfg = synth.ModelConfig(family=synth.LLAMA, n_layers=4, d_model=256, n_heads=8, head_dim=32, d_ffn=1024, vocab=1000,
                            dtype="bf16", hsm_m1=512, hsm_m2=1024, max_batch=1, max_seq=P, max_pass_tokens=P)
    m = adept.Model(cfg, synth.make_weights(cfg, seed=150))
    tok = synth.make_tokens(151, 1, P, cfg.vocab).cuda()
    exits = torch.full((1, P), 4, dtype=torch.int32, device="cuda")

    def best():
        t = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            m.prefill(tok, 0.9, exits)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        return min(t)

    early = best()
    adept.adept_set_option(m.h, adept.OPT_PROFILE, 1)
    apart = best()
    m.check()
    m.close()
    assert early < 1.15 * apart, (early, apart)
