"""The weight-streaming tcgen05 GEMM (9 to 128 token rows) against the oracle: row counts at the edges of its
16-row operand boxes and 32-token epilogue blocks, K of an odd number of 64-k chunks, outputs that are no multiple of
its 128-feature tile (a ragged vocabulary among them), tiles split over many CTAs, layers with no rows left, and
grouped fills of several layers."""
import numpy as np
import pytest
import torch

import synth
from oracle import adept_oracle as O
from parity_utils import Pair, assert_rows_close, compare_decode, compare_prefill

import paper_2601_03700_gb300 as adept

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    adept.load_library()


def config(family, B, P, **kw):
    base = dict(family=family, n_layers=5, d_model=320, n_heads=5, head_dim=64, d_ffn=448, vocab=1003, max_pos=256,
                n_classes=3 if family == synth.BERT else 0, dtype="bf16", hsm_m1=576, hsm_m2=1088, max_batch=B,
                max_seq=max(P + 4, 16), max_pass_tokens=max(B * P, B), block_shuffle_seed=5)
    base.update(kw)
    return synth.ModelConfig(**base)


@pytest.mark.parametrize("family", [synth.LLAMA, synth.GPT2, synth.BERT])
@pytest.mark.parametrize("B,P", [(9, 1), (1, 16), (1, 17), (3, 11), (2, 40), (1, 127), (8, 16)])
def test_swap_gemm_prompt_matches_oracle(family, B, P):
    pair = Pair(config(family, B, P), seed=90 + P)
    tokens = synth.make_tokens(91, B, P, 1003).numpy()
    forced = synth.forced_exits_uniform(92 + P, B * P, 2, 5).numpy().reshape(B, P)
    compare_prefill(pair, tokens, 0.9, forced)
    compare_prefill(pair, tokens, -2.0)      # every token leaves at layer 2: no rows after it
    pair.close()


@pytest.mark.parametrize("family,B", [(synth.LLAMA, 9), (synth.LLAMA, 16), (synth.GPT2, 16), (synth.GPT2, 33)])
def test_swap_gemm_generation_matches_oracle(family, B):
    pair = Pair(config(family, B, 3), seed=94)
    tokens = synth.make_tokens(95, B, 3, 1003).numpy()
    ores, cache, _ = compare_prefill(pair, tokens, 2.0)
    steps = synth.forced_exits_uniform(96, 4 * B, 2, 5).numpy().reshape(4, B)
    compare_decode(pair, cache, ores.next_token, 4, 0.9, steps)
    pair.compare_cache(cache, B, 7)
    pair.close()


@pytest.mark.parametrize("family", [synth.LLAMA, synth.GPT2])
@pytest.mark.parametrize("B,P", [(9, 1), (1, 45)])
def test_swap_gemm_heads_of_32_match_oracle(family, B, P):
    """One head per 32-feature cell: queries, keys (their rotary halves of 16) and values of the cache epilogue."""
    pair = Pair(config(family, B, P, n_heads=10, n_kv_heads=5, head_dim=32), seed=103)
    tokens = synth.make_tokens(104, B, P, 1003).numpy()
    forced = synth.forced_exits_uniform(105, B * P, 2, 5).numpy().reshape(B, P)
    ores, cache, _ = compare_prefill(pair, tokens, 0.9, forced)
    compare_decode(pair, cache, ores.next_token, 2, 0.9, synth.forced_exits_uniform(106, 2 * B, 2, 5).numpy().reshape(2, B))
    pair.compare_cache(cache, B, P + 2)
    pair.close()


@pytest.mark.parametrize("n", [9, 33, 128])
def test_swap_gemm_grouped_fill_matches_oracle(n):
    cfg = config(synth.LLAMA, 1, 128, n_layers=9)
    pair = Pair(cfg, seed=97)
    adept.adept_seq_reserve(pair.gm.h, [128])
    h = synth.make_mapped_states(98, n, cfg.d_model)
    el = synth.forced_exits_uniform(99, n, 1, 9).numpy()
    pos = np.random.RandomState(3).permutation(128)[:n]
    adept.adept_skip_kv_fill(pair.gm.h, n, h.cuda(), torch.as_tensor(el, dtype=torch.int32).cuda(),
                             torch.zeros(n, dtype=torch.int32, device="cuda"),
                             torch.as_tensor(pos, dtype=torch.int32).cuda())
    pair.gm.check()
    want = O.skip_kv_fill(pair.om, h.double().numpy(), el, pos)
    for r, (k, v, sel) in want.items():
        gk, gv = pair.gpu_kv(r, 0, 128)
        assert_rows_close(gk[pos[sel]], k, pair.tol, f"K layer {r}")
        assert_rows_close(gv[pos[sel]], v, pair.tol, f"V layer {r}")
    pair.close()


def test_swap_gemm_repeats_bit_for_bit():
    cfg = config(synth.LLAMA, 2, 40)
    W = synth.make_weights(cfg, seed=100, device="cuda")
    tok = synth.make_tokens(101, 2, 40, 1003).cuda()
    fz = synth.forced_exits_uniform(102, 80, 2, 5).view(2, 40).cuda()
    m = adept.Model(cfg, W)
    first = m.prefill(tok, 0.9, fz)[1].clone()
    for _ in range(3):
        assert torch.equal(first, m.prefill(tok, 0.9, fz)[1])
    m.check()
    m.close()


def test_waits_running_out_at_any_point_leave_the_clusters_whole():
    """Limits from a few cycles to a few microseconds stop the CTAs of a cluster at different k-blocks (tiles split over up to
    8 CTAs, their rings deeper than a CTA's share and shallower): every pass ends, says so in its status, and the next one is
    right."""
    cfg = config(synth.LLAMA, 2, 30, n_layers=3, d_model=1024, n_heads=16, d_ffn=4096, hsm_m1=2048, hsm_m2=4096)
    pair = Pair(cfg, weights=synth.make_weights(cfg, seed=107, device="cuda"))
    tokens = synth.make_tokens(108, 2, 30, 1003).numpy()
    forced = synth.forced_exits_uniform(109, 60, 2, 3).numpy().reshape(2, 30)
    dev = lambda x: torch.as_tensor(x).cuda()  # noqa: E731
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
