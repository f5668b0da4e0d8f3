"""GPU parity: the CUDA library (through its C ABI) against the CPU oracle on the same
seeded inputs.  Hidden states, logits and KV entries within the row-wise relative
tolerance of the precision contract (1e-4 fp32, 2e-2 bf16); exit layers bit-exact
outside the +-1e-3 similarity band."""
import numpy as np
import pytest
import torch

import synth
from oracle import adept_oracle as O
from parity_utils import Pair, assert_rows_close, compare_decode, compare_prefill, TOL

import paper_2601_03700_gb300 as adept

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    adept.load_library()


def small(family, dtype="bf16", **kw):
    base = dict(family=family, n_layers=6, d_model=256, n_heads=4, head_dim=64, d_ffn=512, vocab=1000,
                max_pos=160, n_classes=2 if family == synth.BERT else 0, dtype=dtype, max_batch=4, max_seq=160,
                hsm_m1=512, hsm_m2=1024)
    if family == synth.BERT:
        base["norm_eps"] = 1e-12
    base.update(kw)
    return synth.ModelConfig(**base)


# --------------------------------------------------------------------------- tiny, fp32

def test_tiny_fp32_threshold_prefill_and_decode():
    """Tiny decoder (4 layers, D=256, 4 heads, SwiGLU 1024, vocab 1024, fp32, seed 0): a
    64-token prompt, then 16 greedy decode steps, cosine threshold 0.95."""
    cfg = synth.tiny_config()
    pair = Pair(cfg, seed=0)
    tokens = synth.make_tokens(0, 1, 64, cfg.vocab).numpy()
    ores, cache, g = compare_prefill(pair, tokens, 0.95)
    compare_decode(pair, cache, ores.next_token, 16, 0.95)
    pair.compare_cache(cache, 1, 64 + 16)
    pair.close()


@pytest.mark.parametrize("delta", [0.2, 0.5, -2.0, float("inf")])
def test_tiny_fp32_thresholds_ragged_batch(delta):
    cfg = synth.tiny_config()
    pair = Pair(cfg, seed=1, std=0.05)
    tokens = synth.make_tokens(1, 3, 37, cfg.vocab).numpy()
    ores, cache, g = compare_prefill(pair, tokens, delta)
    if delta == -2.0:
        assert np.all(g["exit"] == 2)
    if delta == float("inf"):
        assert np.all(g["exit"] == cfg.n_layers)
    compare_decode(pair, cache, ores.next_token, 3, delta)
    pair.close()


def test_tiny_fp32_forced_exits_and_hsm_identity():
    cfg = synth.tiny_config(n_layers=6)
    pair = Pair(cfg, seed=2, std=0.05)
    tokens = synth.make_tokens(2, 2, 45, cfg.vocab).numpy()
    forced = synth.forced_exits_uniform(2, 90, 2, 6).numpy().reshape(2, 45)
    for ident in (False, True):
        ores, cache, g = compare_prefill(pair, tokens, 0.5, forced, hsm_identity=ident)
        fsteps = synth.forced_exits_uniform(3, 8, 2, 6).numpy().reshape(4, 2)
        compare_decode(pair, cache, ores.next_token, 4, 0.5, fsteps, hsm_identity=ident)
        pair.compare_cache(cache, 2, 45 + 4)
    pair.close()


# --------------------------------------------------------------------------- bf16 families

@pytest.mark.parametrize("family", [synth.LLAMA, synth.GPT2, synth.BERT, "llama_gqa"])
def test_bf16_families_forced(family):
    if family == "llama_gqa":   # grouped-query attention: 4 query heads share 2 KV heads
        family, kw = synth.LLAMA, dict(n_heads=4, n_kv_heads=2, head_dim=64)
    else:
        kw = dict(n_heads=2, head_dim=128) if family == synth.LLAMA else {}
    cfg = small(family, **kw)
    pair = Pair(cfg, seed=3)
    B, P = 3, 70
    tokens = synth.make_tokens(3, B, P, cfg.vocab).numpy()
    forced = synth.forced_exits_uniform(4, B * P, 2, cfg.n_layers).numpy().reshape(B, P)
    ores, cache, g = compare_prefill(pair, tokens, 0.9, forced)
    if family != synth.BERT:
        fsteps = synth.forced_exits_uniform(5, 5 * B, 2, cfg.n_layers).numpy().reshape(5, B)
        compare_decode(pair, cache, ores.next_token, 5, 0.9, fsteps)
        pair.compare_cache(cache, B, P + 5)
    pair.close()


@pytest.mark.parametrize("family", [synth.LLAMA, synth.GPT2, synth.BERT])
def test_bf16_families_threshold(family):
    cfg = small(family)
    pair = Pair(cfg, seed=6, std=0.05)
    tokens = synth.make_tokens(6, 2, 50, cfg.vocab).numpy()
    for delta in (0.9, 0.6):
        ores, cache, g = compare_prefill(pair, tokens, delta)
        if family != synth.BERT:
            compare_decode(pair, cache, ores.next_token, 3, delta)
    pair.close()


# --------------------------------------------------------------------------- skipped-layer fill ABI

@pytest.mark.parametrize("dtype,n", [("f32", 150), ("bf16", 150), ("bf16", 7)])
def test_skip_kv_fill_matches_oracle(dtype, n):
    """adept_skip_kv_fill: every (token, r > i*) entry equals layer r's K/V projection of s~
    (7 bf16 tokens take the grouped weight-streaming launch, 150 the grouped tcgen05 GEMM)."""
    cfg = small(synth.LLAMA, dtype=dtype, n_layers=8, n_heads=2, head_dim=128, block_shuffle_seed=7)
    pair = Pair(cfg, seed=8)
    lens = [cfg.max_seq] * cfg.max_batch
    adept.adept_seq_reserve(pair.gm.h, lens)
    h = synth.make_mapped_states(9, n, cfg.d_model, dtype=cfg.torch_dtype)
    el = synth.forced_exits_uniform(10, n, 1, cfg.n_layers).numpy()
    seq = synth.randint(11, "seq", n, 0, cfg.max_batch - 1).numpy()
    # distinct positions per sequence
    pos = np.zeros(n, dtype=np.int64)
    for b in range(cfg.max_batch):
        idx = np.nonzero(seq == b)[0]
        pos[idx] = synth.randint(12 + b, "perm", 1, 0, 0).numpy()[0] + np.arange(len(idx))
    adept.adept_skip_kv_fill(pair.gm.h, n, h.cuda().contiguous(), torch.as_tensor(el, dtype=torch.int32).cuda(),
                             torch.as_tensor(seq, dtype=torch.int32).cuda(), torch.as_tensor(pos, dtype=torch.int32).cuda())
    pair.gm.check()
    ref = O.skip_kv_fill(pair.om, h.double().numpy(), el, pos)
    checked = 0
    for r, (k, v, sel) in ref.items():
        for b in range(cfg.max_batch):
            rows = sel[seq[sel] == b]
            if len(rows) == 0:
                continue
            gk, gv = pair.gpu_kv(r, b, cfg.max_seq)
            assert_rows_close(gk[pos[rows]], k[np.searchsorted(sel, rows)], pair.tol, f"K r={r}")
            assert_rows_close(gv[pos[rows]], v[np.searchsorted(sel, rows)], pair.tol, f"V r={r}")
            checked += len(rows)
    assert checked >= n - int(np.sum(el == cfg.n_layers))
    pair.close()


# --------------------------------------------------------------------------- error paths

def test_device_input_errors_are_reported():
    cfg = synth.tiny_config()
    pair = Pair(cfg, seed=0)
    tk = torch.zeros(1, 8, dtype=torch.int32, device="cuda")
    bad = torch.ones(1, 8, dtype=torch.int32, device="cuda")      # forced layer 1 is not eligible
    pair.gm.prefill(tk, 0.5, bad)
    with pytest.raises(adept.AdeptError) as ei:
        pair.gm.check()
    assert ei.value.status == 6
    tk2 = torch.full((1, 8), cfg.vocab + 5, dtype=torch.int32, device="cuda")
    pair.gm.prefill(tk2, 0.5)
    with pytest.raises(adept.AdeptError):
        pair.gm.check()
    pair.gm.check()  # cleared
    with pytest.raises(adept.AdeptError) as ei:
        pair.gm.prefill(torch.zeros(9, 8, dtype=torch.int32, device="cuda"), 0.5)
    assert ei.value.status == 3
    pair.close()


def test_synth_generator_cpu_and_cuda_agree():
    a = synth.normal(5, "w", (3, 100003), std=0.02, dtype=torch.bfloat16)
    b = synth.normal(5, "w", (3, 100003), std=0.02, dtype=torch.bfloat16, device="cuda").cpu()
    assert torch.equal(a.view(torch.int16), b.view(torch.int16))


def test_prompt_pass_mapper_split_by_live_rows():
    """The prompt pass's mapper products at device-side exit counts near and far below their
    bound: 600 tokens with 300 leaving at layer 2 and 100 at layers 3 and 4 (the paired tiles
    take their width from the count; a D = 512 model with mapper widths 2048 / 4096, so that
    the counts lie on both sides of a change of width)."""
    cfg = small(synth.GPT2, n_layers=6, d_model=512, n_heads=8, head_dim=64, d_ffn=1024, hsm_m1=2048, hsm_m2=4096,
                max_seq=160, max_pos=160)
    pair = Pair(cfg, seed=12, std=0.04)
    B, P = 4, 150
    tokens = synth.make_tokens(12, B, P, cfg.vocab).numpy()
    law = np.array([2] * 300 + [3] * 100 + [4] * 100 + [6] * 100)
    rng = np.random.default_rng(12)
    forced = rng.permutation(law).reshape(B, P)
    compare_prefill(pair, tokens, 0.9, forced)
    pair.close()


def test_tensor_core_gemm_matches_simt_gemm():
    """The tcgen05 grouped GEMM and the SIMT GEMM give the same pass (bf16 noise level),
    on a shape with ragged M tiles (130-token prompts) and every epilogue kind."""
    from parity_utils import row_rel_err
    for family, kw in ((synth.LLAMA, dict(n_heads=2, head_dim=128)), (synth.GPT2, {}), (synth.BERT, {})):
        cfg = small(family, n_layers=4, max_seq=256, max_pos=256, **kw)
        W = synth.make_weights(cfg, seed=0)
        m = adept.Model(cfg, W)
        tokens = synth.make_tokens(0, 2, 130, cfg.vocab).cuda()
        forced = synth.forced_exits_uniform(0, 260, 2, 4).view(2, 130).cuda()
        out = {}
        for simt in (1, 0):
            adept.adept_set_option(m.h, adept.OPT_GEMM_SIMT, simt)
            ex, lg, nx, sim = m.prefill(tokens, 0.5, forced)
            m.check()
            out[simt] = (ex.cpu().numpy(), m.final_states(260).cpu().numpy(), lg.cpu().numpy(),
                         m.read_kv(1, 1, 0, 130)[0].float().cpu().numpy())
        np.testing.assert_array_equal(out[0][0], out[1][0])
        assert row_rel_err(out[0][3], out[1][3]).max() < 2e-3      # first layer's K: one GEMM
        assert row_rel_err(out[0][1], out[1][1]).max() < 2e-2
        assert row_rel_err(out[0][2], out[1][2]).max() < 2e-2
        m.close()


def test_decode_graph_replay_equals_direct_launches():
    """A captured generation step replays to the same bits as direct launches."""
    cfg = small(synth.GPT2, n_layers=6)
    W = synth.make_weights(cfg, seed=21)
    outs = []
    for graph in (0, 1):
        m = adept.Model(cfg, W)
        adept.adept_set_option(m.h, adept.OPT_DECODE_GRAPH, graph)
        tokens = synth.make_tokens(21, 3, 40, cfg.vocab).cuda()
        ex, lg, nx, _ = m.prefill(tokens, 0.5, synth.forced_exits_uniform(21, 120, 2, 6).view(3, 40).cuda())
        steps = []
        fs = synth.forced_exits_uniform(22, 18, 2, 6).view(6, 3).cuda()
        for s in range(6):
            ex, lg, nx, sim = m.decode_step(nx, 0.5, fs[s] if s % 2 == 0 else None)
            steps.append((ex.cpu(), lg.cpu(), nx.cpu(), sim.cpu()))
        m.check()
        outs.append((steps, m.read_kv(6, 1, 0, 46)[0].float().cpu()))
        m.close()
    for a, b in zip(outs[0][0], outs[1][0]):
        for x, y in zip(a, b):
            assert torch.equal(x.nan_to_num(7.0), y.nan_to_num(7.0))
    assert torch.equal(outs[0][1], outs[1][1])


def test_generation_step_gemm_matches_tensor_core_gemm():
    """The generation-step GEMM (weight streaming, K-split clusters, fused input
    standardisation) against the tcgen05 path with separate standardisation launches: the
    same exits, logits and cache entries at bf16 noise level, for 3 (one 8-token block)
    and 12 (two blocks) sequences, ragged output tiles (vocab 1000) and every epilogue
    of the decoders.  Both runs are fed the same tokens each step (a greedy choice can differ
    between two correct runs where the top two logits are within rounding of each other)."""
    from parity_utils import row_rel_err
    for family, kw in ((synth.LLAMA, dict(n_heads=2, head_dim=128)), (synth.GPT2, {})):
        for B in (3, 12):
            cfg = small(family, n_layers=5, max_batch=B, **kw)
            W = synth.make_weights(cfg, seed=31)
            out = {}
            for dg in (1, 0):
                m = adept.Model(cfg, W)
                adept.adept_set_option(m.h, adept.OPT_DECODE_GEMM, dg)
                tokens = synth.make_tokens(31, B, 20, cfg.vocab).cuda()
                forced = synth.forced_exits_uniform(31, B * 20, 2, 5).view(B, 20).cuda()
                ex, lg, nx, _ = m.prefill(tokens, 0.5, forced)
                steps = []
                fs = synth.forced_exits_uniform(32, 4 * B, 2, 5).view(4, B).cuda()
                ts = synth.make_tokens(33, 4, B, cfg.vocab).cuda()
                for s in range(4):
                    ex, lg, nx, sim = m.decode_step(ts[s].contiguous(), 0.5, fs[s])
                    steps.append((ex.cpu().numpy(), lg.cpu().numpy(), m.final_states(B).cpu().numpy()))
                m.check()
                out[dg] = (steps, m.read_kv(4, B - 1, 0, 24)[0].float().cpu().numpy())
                m.close()
            for a, b in zip(out[0][0], out[1][0]):
                np.testing.assert_array_equal(a[0], b[0])
                assert row_rel_err(a[1], b[1]).max() < 2e-2
                assert row_rel_err(a[2], b[2]).max() < 2e-2
            assert row_rel_err(out[0][1], out[1][1]).max() < 2e-2


# --------------------------------------------------------------------------- threshold calibration

@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_threshold_calibration_matches_oracle(dtype):
    """adept_calibrate_threshold (bisection on delta over device prompt passes) against the
    oracle's calibration on the same model and batch: the same thresholds pass for pass
    while no similarity of the batch falls within the +-1e-3 band of the threshold tried,
    the target reached on both sides, and the oracle's RDC at the device's delta."""
    from parity_utils import BAND
    cfg = synth.tiny_config(n_layers=6) if dtype == "f32" else small(synth.GPT2, n_layers=6)
    pair = Pair(cfg, seed=44, std=0.05)
    B, P = 2, 24
    tokens = synth.make_tokens(44, B, P, cfg.vocab)
    grid = np.linspace(-1.0, 1.0, 21)
    scan = [O.reduction_in_computation(O.prefill(pair.om, O.OracleCache(cfg, B, P), tokens.numpy(), d).exit_layer,
                                       cfg.n_layers) for d in grid]
    mids = sorted({r for r in scan if 0.0 < r < 1 - 2 / cfg.n_layers})
    assert mids
    target, tol = mids[len(mids) // 2], 0.02
    d_o, r_o, hist = O.calibrate_threshold(pair.om, tokens.numpy(), target, tol=tol, max_iter=16)
    d_g, r_g, n_g = adept.adept_calibrate_threshold(pair.gm.h, B, P, tokens.cuda().view(-1), target, tol, 16)
    pair.gm.check()
    assert abs(r_o - target) <= tol and abs(r_g - target) <= tol + 1e-6
    # pass for pass: identical thresholds unless a similarity sat in the band of one tried
    banded = False
    for dd, _ in hist:
        res = O.prefill(pair.om, O.OracleCache(cfg, B, P), tokens.numpy(), dd)
        with np.errstate(invalid="ignore"):
            banded |= bool(np.any(np.abs(res.sim - dd) <= BAND))
    if not banded:
        assert n_g == len(hist) and np.float32(d_g) == np.float32(d_o)
    # the device's threshold gives the oracle the device's reduction (decisions agree)
    res = O.prefill(pair.om, O.OracleCache(cfg, B, P), tokens.numpy(), d_g)
    with np.errstate(invalid="ignore"):
        if not np.any(np.abs(res.sim - d_g) <= BAND):
            assert O.reduction_in_computation(res.exit_layer, cfg.n_layers) == pytest.approx(r_g, abs=1e-6)
    pair.close()


# --------------------------------------------------------------------------- exit-rule variants

@pytest.mark.parametrize("metric", ["local", "both"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_exit_metric_variants_match_oracle(metric, dtype):
    """Local similarity cos(s_i, s_{i-1}) and both similarities (App. H.3): prompt pass and
    generation steps against the oracle, thresholds that leave some tokens early."""
    cfg = synth.tiny_config(n_layers=6) if dtype == "f32" else small(synth.LLAMA, n_heads=2, head_dim=128)
    pair = Pair(cfg, seed=61, std=0.05)
    tokens = synth.make_tokens(61, 2, 30, cfg.vocab).numpy()
    probe = O.prefill(pair.om, O.OracleCache(cfg, 2, 32), tokens, np.inf, metric=metric).sim
    delta = float(np.nanquantile(probe, 0.7))
    ores, cache, g = compare_prefill(pair, tokens, delta, metric=metric)
    assert 2 <= ores.exit_layer.min() and ores.exit_layer.min() < cfg.n_layers
    compare_decode(pair, cache, ores.next_token, 3, delta, metric=metric)
    pair.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_all_at_once_prompt_exits_match_oracle(dtype):
    """All-at-once prompt exits (App. H.2): every token of a sequence leaves with its last
    prompt token; exits, final states, logits and the cache against the oracle."""
    cfg = synth.tiny_config(n_layers=6) if dtype == "f32" else small(synth.GPT2)
    pair = Pair(cfg, seed=62, std=0.05)
    B, P = 3, 20
    tokens = synth.make_tokens(62, B, P, cfg.vocab).numpy()
    probe = O.prefill(pair.om, O.OracleCache(cfg, B, P), tokens, np.inf).sim.reshape(B, P, -1)[:, P - 1]
    delta = float(np.nanquantile(probe, 0.6))
    ores, cache, g = compare_prefill(pair, tokens, delta, all_at_once=True)
    ex = g["exit"].reshape(B, P)
    assert np.all(ex == ex[:, -1:])
    pair.close()


def test_encoder_stop_entirely_matches_oracle():
    """Encoder "stop entirely" (Sec. 4.3, downstream tasks): forced and threshold exits,
    exited tokens left out of deeper attention and given no deeper K/V; final states,
    classifier logits and every K/V the oracle wrote, against the oracle."""
    from parity_utils import assert_rows_close
    cfg = small(synth.BERT)
    pair = Pair(cfg, seed=63)
    B, P = 3, 40
    tokens = synth.make_tokens(63, B, P, cfg.vocab).numpy()
    forced = synth.forced_exits_uniform(63, B * P, 2, cfg.n_layers).numpy().reshape(B, P)
    for fz, delta in ((forced, 0.9), (None, 0.6)):
        ores, cache, g = compare_prefill(pair, tokens, delta, fz, check_cache=False, stop_entirely=True)
        for l in range(1, cfg.n_layers + 1):
            for b in range(B):
                k, v = pair.gpu_kv(l, b, P)
                ok = ~np.isnan(cache.K[l - 1][b, :P, 0, 0])   # written by the oracle: tokens active at l
                if l == 1:
                    assert ok.all()
                if not ok.any():
                    continue
                assert_rows_close(k[ok], cache.K[l - 1][b, :P][ok], pair.tol, f"K layer {l} seq {b}")
                assert_rows_close(v[ok], cache.V[l - 1][b, :P][ok], pair.tol, f"V layer {l} seq {b}")
    adept.adept_set_option(pair.gm.h, adept.OPT_STOP_ENTIRELY, 0)
    pair.close()


@pytest.mark.parametrize("B,P", [(3, 40), (1, 240)])
def test_encoder_stop_entirely_with_heads_of_32(B, P):
    """The key mask in the attention of heads of 32, keys in several blocks of 32, whole blocks of them gone."""
    cfg = small(synth.BERT, n_layers=6, n_heads=8, n_kv_heads=4, head_dim=32, n_classes=2, max_pos=P, max_seq=P,
                max_batch=B)
    pair = Pair(cfg, seed=31)
    tokens = synth.make_tokens(31, B, P, cfg.vocab).numpy()
    mixed = synth.forced_exits_uniform(32, B * P, 2, 6).numpy().reshape(B, P)
    blocks = np.where(np.arange(P)[None, :] // 32 % 2 == 0, 2, mixed)   # whole blocks gone after layer 2
    for forced in (mixed, blocks):
        compare_prefill(pair, tokens, 0.9, forced, check_cache=False, stop_entirely=True)
    pair.close()
