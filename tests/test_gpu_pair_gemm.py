"""The paired tcgen05 GEMM (more than 128 token rows) against the oracle: row counts at the edges of its 256-row tiles and
of its CTAs' 128-row halves, inner sizes that are no multiple of its 64-wide k-blocks or of whole tiles, live row counts from
none to all (which move its tile width), grouped fills of many layers, and the logits of a ragged vocabulary."""
import numpy as np
import pytest
import torch

import synth
from oracle import adept_oracle as O
from parity_utils import Pair, assert_rows_close, compare_prefill

import paper_2601_03700_gb300 as adept

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    adept.load_library()


def config(family, B, P, **kw):
    base = dict(family=family, n_layers=5, d_model=320, n_heads=5, head_dim=64, d_ffn=464, vocab=1003, max_pos=320,
                n_classes=3 if family == synth.BERT else 0, dtype="bf16", hsm_m1=584, hsm_m2=1096, max_batch=B,
                max_seq=max(P + 4, 16), max_pass_tokens=max(B * P, B), block_shuffle_seed=5)
    base.update(kw)
    return synth.ModelConfig(**base)


@pytest.mark.parametrize("family", [synth.LLAMA, synth.GPT2, synth.BERT])
@pytest.mark.parametrize("B,P", [(1, 129), (5, 51), (1, 257), (3, 128), (131, 4)])
def test_pair_gemm_prompt_matches_oracle(family, B, P):
    pair = Pair(config(family, B, P), seed=110 + P)
    tokens = synth.make_tokens(111, B, P, 1003).numpy()
    forced = synth.forced_exits_uniform(112 + P, B * P, 2, 5).numpy().reshape(B, P)
    compare_prefill(pair, tokens, 0.9, forced)
    compare_prefill(pair, tokens, -2.0)      # every token leaves at layer 2: no rows after it
    pair.close()


@pytest.mark.parametrize("family", [synth.LLAMA, synth.GPT2])
def test_pair_gemm_heads_of_32_match_oracle(family):
    """One head per 32-column chunk: queries, keys (their rotary halves of 16) and values of the cache epilogue."""
    pair = Pair(config(family, 1, 141, n_heads=10, n_kv_heads=5, head_dim=32), seed=126)
    tokens = synth.make_tokens(127, 1, 141, 1003).numpy()
    forced = synth.forced_exits_uniform(128, 141, 2, 5).numpy().reshape(1, 141)
    _, cache, _ = compare_prefill(pair, tokens, 0.9, forced)
    pair.compare_cache(cache, 1, 141)
    pair.close()


@pytest.mark.parametrize("n", [129, 300])
def test_pair_gemm_grouped_fill_matches_oracle(n):
    cfg = config(synth.LLAMA, 1, 300, n_layers=9)
    pair = Pair(cfg, seed=117)
    adept.adept_seq_reserve(pair.gm.h, [300])
    h = synth.make_mapped_states(118, n, cfg.d_model)
    el = synth.forced_exits_uniform(119, n, 1, 9).numpy()
    pos = np.random.RandomState(3).permutation(300)[:n]
    adept.adept_skip_kv_fill(pair.gm.h, n, h.cuda(), torch.as_tensor(el, dtype=torch.int32).cuda(),
                             torch.zeros(n, dtype=torch.int32, device="cuda"),
                             torch.as_tensor(pos, dtype=torch.int32).cuda())
    pair.gm.check()
    want = O.skip_kv_fill(pair.om, h.double().numpy(), el, pos)
    for r, (k, v, sel) in want.items():
        gk, gv = pair.gpu_kv(r, 0, 300)
        assert_rows_close(gk[pos[sel]], k, pair.tol, f"K layer {r}")
        assert_rows_close(gv[pos[sel]], v, pair.tol, f"V layer {r}")
    pair.close()


def test_short_wait_limit_times_out_and_recovers():
    """Waits that run out in a pass on the paired tiles: the status says so, the context stays usable, and with the limit
    restored the same model matches the oracle."""
    pair = Pair(config(synth.GPT2, 2, 150), seed=120)
    tokens = synth.make_tokens(121, 2, 150, 1003).numpy()
    forced = synth.forced_exits_uniform(122, 300, 2, 5).numpy().reshape(2, 150)
    adept.adept_set_wait_limit(32)
    try:
        pair.gm.prefill(torch.as_tensor(tokens).cuda(), 0.9, torch.as_tensor(forced).cuda())
        with pytest.raises(adept.AdeptError) as ei:
            pair.gm.check()
        assert ei.value.status == 5, str(ei.value)
    finally:
        adept.adept_set_wait_limit(0)
    compare_prefill(pair, tokens, 0.9, forced)
    pair.close()


def test_waits_running_out_at_any_point_leave_the_pair_whole():
    """Limits from a few cycles to a few microseconds stop the CTAs of a pair at different k-blocks, each with copies under
    way that the other has not matched: every pass ends, says so in its status, and the next one is right."""
    cfg = config(synth.GPT2, 3, 200, n_layers=3, d_model=1024, n_heads=16, d_ffn=4096, hsm_m1=2048, hsm_m2=4096)
    pair = Pair(cfg, weights=synth.make_weights(cfg, seed=123, device="cuda"))
    tokens = synth.make_tokens(124, 3, 200, 1003).numpy()
    forced = synth.forced_exits_uniform(125, 600, 2, 3).numpy().reshape(3, 200)
    dev = lambda x: torch.as_tensor(x).cuda()  # noqa: E731
    pair.gm.prefill(dev(tokens), 0.9, dev(forced))
    pair.gm.check()
    stopped = 0
    for limit in (1, 32, 200, 500, 1000, 1500, 2000, 3000, 5000, 10000):
        adept.adept_set_wait_limit(limit)
        try:
            pair.gm.prefill(dev(tokens), 0.9, dev(forced))
            try:
                pair.gm.check()
            except adept.AdeptError as e:
                assert e.status == 5, str(e)
                stopped += 1
        finally:
            adept.adept_set_wait_limit(0)
    assert stopped >= 2
    compare_prefill(pair, tokens, 0.9, forced)
    pair.close()
