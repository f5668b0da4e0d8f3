"""The last launch of a generation step: greedy tokens (the first of equal logits) and the copies of logits, exits and
similarities, for vocabularies in one part and in many, over repeated steps and with outputs left out; logits that are NaN."""
import pytest
import torch

import synth

import paper_2601_03700_gb300 as adept

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab", [1000, 4097, 50257])
@pytest.mark.parametrize("batch", [1, 5])
def test_step_outputs(vocab, batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = synth.ModelConfig(family=synth.GPT2, n_layers=3, d_model=128, n_heads=2, head_dim=64, d_ffn=256, vocab=vocab,
                            max_pos=64, dtype="bf16", hsm_m1=256, hsm_m2=512, max_batch=batch, max_seq=32,
                            max_pass_tokens=4 * batch)
    W = synth.make_weights(cfg, seed=140, device="cuda")
    W["tok_emb"][vocab // 2:] = W["tok_emb"][:vocab - vocab // 2].clone()   # equal rows: equal logits (tied head)
    m = adept.Model(cfg, W)
    m.prefill(synth.make_tokens(141, batch, 4, vocab).cuda(), 0.9)
    tok = torch.zeros(batch, dtype=torch.int32, device="cuda")
    for step in range(4):
        ex, lg, nx, sims = m.decode_step(tok, 0.9)
        want = (lg == lg.max(dim=1, keepdim=True).values).int().argmax(dim=1)
        assert torch.equal(nx.long(), want)
        assert int(ex.min()) >= 2 and int(ex.max()) <= 3 and sims.shape == (batch, 3)
        adept.adept_decode_step(m.h, batch, tok, 0.9, next_token_out=nx)   # the others left out
        tok = nx.clone()
    m.check()
    m.close()


@pytest.mark.parametrize("vocab", [1000, 4097])
def test_nan_logits_are_never_the_token(vocab):
    """A NaN logit is passed over, at a part's first and last column too; a row of nothing else gives token 0."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = synth.ModelConfig(family=synth.LLAMA, n_layers=3, d_model=128, n_heads=2, head_dim=64, d_ffn=256, vocab=vocab,
                            dtype="bf16", hsm_m1=256, hsm_m2=512, max_batch=3, max_seq=32, max_pass_tokens=12)
    W = synth.make_weights(cfg, seed=142, device="cuda")
    tok = synth.make_tokens(143, 3, 4, vocab).cuda()
    for bad in ([0, 129, vocab // 2, vocab - 1], list(range(vocab))):
        head = W["lm_head"].clone()
        head[bad] = float("nan")
        m = adept.Model(cfg, {**W, "lm_head": head})
        nx = m.prefill(tok, 0.9)[2]
        for _ in range(3):   # launched directly, captured, replayed
            _, lg, nx, _ = m.decode_step(nx.clone(), 0.9)
            assert torch.isnan(lg[:, bad]).all() and int(torch.isnan(lg).sum()) == 3 * len(bad)
            lg = lg.masked_fill(torch.isnan(lg), float("-inf"))
            assert torch.equal(nx.long(), (lg == lg.max(dim=1, keepdim=True).values).int().argmax(dim=1))
        m.check()
        m.close()


def test_final_states_of_a_replayed_step():
    """The rows that may be read after a step are that step's, also when it is replayed after steps of another batch."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = synth.ModelConfig(family=synth.GPT2, n_layers=3, d_model=128, n_heads=2, head_dim=64, d_ffn=256, vocab=500,
                            max_pos=64, dtype="bf16", hsm_m1=256, hsm_m2=512, max_batch=5, max_seq=32, max_pass_tokens=20)
    m = adept.Model(cfg, synth.make_weights(cfg, seed=144, device="cuda"))
    m.prefill(synth.make_tokens(145, 5, 4, cfg.vocab).cuda(), 0.9)
    for batch in (5, 5, 5, 2, 2, 5, 2, 5):   # each launched directly, captured, replayed
        m.decode_step(torch.arange(batch, dtype=torch.int32, device="cuda"), 0.9)
        assert torch.isfinite(m.final_states(batch)).all()
        with pytest.raises(adept.AdeptError):
            m.final_states(batch + 1)
    m.check()
    m.close()
