"""The work that a program has this framework do, as measurable cases.

A case is a model of one of the repository's shapes and one call sequence on it: a decoder's
turn (prompt pass and generation steps), an encoder's pass, an encoder-decoder's turn, a
skipped-layer K/V fill, or a training step of the hidden-state mapper.  Sizes are those of the
repository's configurations and benchmark; models of the Llama-2-7B shape carry 4 or 8 of its 32
equal layers, so that a case is a block of layers and not a whole model's rounding history.
The mapper's exits are forced from a law (as the benchmark forces them) wherever a rounding
step could move a token's exit layer; the fp32 model decides by its threshold.  Generation
steps are fed given tokens, as a program that scores or verifies a continuation feeds them.
"""
import math
from types import SimpleNamespace

import torch

import paper_2601_03700_gb300 as adept

MAPPER = ["hsm.g0", "hsm.conv_w", "hsm.conv_b", "hsm.fc1_w", "hsm.fc1_b", "hsm.fc2_w", "hsm.fc2_b", "hsm.fc3_w",
          "hsm.fc3_b", "hsm.g1", "hsm.fc4_w", "hsm.fc4_b", "hsm.g2"]

#: Model shapes, by the names the repository's configurations give them.
SHAPES = {
    "tiny": dict(family="llama", d_model=256, n_heads=4, head_dim=64, d_ffn=1024, vocab=1024, dtype="f32", max_seq=128),
    "gpt2_small": dict(family="gpt2", d_model=768, n_heads=12, head_dim=64, d_ffn=3072, vocab=50257, max_pos=1024,
                       max_seq=1024),
    "llama7b": dict(family="llama", d_model=4096, n_heads=32, head_dim=128, d_ffn=11008, vocab=32000, hsm_m1=8192,
                    hsm_m2=32768, max_seq=2304),
    "llama7b_gqa": dict(family="llama", d_model=4096, n_heads=32, n_kv_heads=8, head_dim=128, d_ffn=11008, vocab=32000,
                        hsm_m1=8192, hsm_m2=32768, max_seq=512),
    # the fill reads the K/V projections alone: the other weights are narrow, to be quick to make
    "llama7b_kv": dict(family="llama", d_model=4096, n_heads=32, head_dim=128, d_ffn=1024, vocab=1024, hsm_m1=1024,
                       hsm_m2=1024, max_seq=2304),
    "bert_base": dict(family="bert", d_model=768, n_heads=12, head_dim=64, d_ffn=3072, vocab=30522, max_pos=512,
                      n_classes=2, norm_eps=1e-12, max_seq=128),
    "ofa_enc": dict(family="bert", d_model=768, n_heads=12, head_dim=64, d_ffn=3072, vocab=50265, max_pos=1024,
                    n_classes=3, max_seq=256),
    "ofa_dec": dict(family="gpt2", d_model=768, n_heads=12, head_dim=64, d_ffn=3072, vocab=50265, max_pos=1024,
                    max_seq=32),
}


def listed():
    return [
        # the first workload of the benchmark's configurations: fp32, a 64-token prompt and 16 steps, where
        # launches and latency are all there is
        dict(name="tiny_fp32_turn", kind="turn", shape="tiny", layers=4, batch=1, prompt=64, steps=16, lo=0, hi=0),
        # one user of a small decoder: a short prompt, then token by token
        dict(name="gpt2_turn_b1", kind="turn", shape="gpt2_small", layers=12, batch=1, prompt=33, steps=16, lo=4, hi=12),
        # the benchmark's GPT-2-small workload with a part of its steps
        dict(name="gpt2_turn_b8", kind="turn", shape="gpt2_small", layers=12, batch=8, prompt=512, steps=8, lo=4, hi=12),
        # one user of a large decoder: generation is a stream of weights
        dict(name="llama_turn_b1", kind="turn", shape="llama7b", layers=8, batch=1, prompt=77, steps=12, lo=3, hi=8),
        # a long prompt of a large decoder (the headline's 2048 tokens)
        dict(name="llama_prompt", kind="turn", shape="llama7b", layers=4, batch=1, prompt=2048, steps=0, lo=2, hi=4),
        # several users of a grouped-query decoder at once
        dict(name="llama_gqa_turn_b16", kind="turn", shape="llama7b_gqa", layers=4, batch=16, prompt=150, steps=6, lo=2,
             hi=4),
        # the benchmark's encoder batch: 64 sentences of 128 tokens
        dict(name="bert_encode_64x128", kind="turn", shape="bert_base", layers=12, batch=64, prompt=128, steps=0, lo=4,
             hi=12),
        # the benchmark's encoder-decoder: 8 sources of 256 tokens, an 8-token target prompt, steps
        dict(name="ofa_turn_b8", kind="encdec", layers=6, batch=8, source=256, prompt=8, steps=8, lo=2, hi=6),
        # K/V of a few exited tokens (what a generation step leaves behind)
        dict(name="fill_7", kind="fill", shape="llama7b_kv", layers=8, tokens=7),
        # K/V of a prompt's exited tokens
        dict(name="fill_2000", kind="fill", shape="llama7b_kv", layers=8, tokens=2000),
        # mapper training: 64 sequences x 64 exited tokens of a decoder; an encoder's with its [CLS] rows
        dict(name="train_gpt2_4096", kind="train", shape="gpt2_small", layers=1, rows=4096),
        dict(name="train_bert_1000", kind="train", shape="bert_base", layers=1, rows=1000),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["tiny", "gpt2", "gpt2", "llama", "prompt", "gqa", "bert", "bert", "ofa", "fill", "fill", "train"])
    if kind == "tiny":
        return dict(kind="turn", shape="tiny", layers=4, batch=rng.randint(1, 4), prompt=_log_int(rng, 1, 96),
                    steps=rng.randint(0, 16), lo=0, hi=0)
    if kind == "gpt2":
        return dict(kind="turn", shape="gpt2_small", layers=12, batch=rng.randint(1, 8), prompt=_log_int(rng, 1, 512),
                    steps=rng.randint(1, 16), lo=rng.randint(2, 8), hi=12)
    if kind == "llama":
        return dict(kind="turn", shape="llama7b", layers=8, batch=rng.randint(1, 4), prompt=_log_int(rng, 1, 256),
                    steps=rng.randint(2, 12), lo=rng.randint(2, 6), hi=8)
    if kind == "prompt":
        return dict(kind="turn", shape="llama7b", layers=4, batch=1, prompt=_log_int(rng, 64, 2048), steps=0, lo=2, hi=4)
    if kind == "gqa":
        return dict(kind="turn", shape="llama7b_gqa", layers=4, batch=_log_int(rng, 1, 16), prompt=_log_int(rng, 1, 150),
                    steps=rng.randint(1, 6), lo=2, hi=4)
    if kind == "bert":
        return dict(kind="turn", shape="bert_base", layers=12, batch=_log_int(rng, 1, 64), prompt=_log_int(rng, 4, 128),
                    steps=0, lo=rng.randint(2, 8), hi=12)
    if kind == "ofa":
        return dict(kind="encdec", layers=6, batch=rng.randint(1, 8), source=_log_int(rng, 8, 256),
                    prompt=rng.randint(1, 16), steps=rng.randint(1, 8), lo=2, hi=6)
    if kind == "fill":
        return dict(kind="fill", shape="llama7b_kv", layers=8, tokens=_log_int(rng, 1, 2000))
    return dict(kind="train", shape=rng.choice(["gpt2_small", "bert_base"]), layers=1, rows=_log_int(rng, 16, 4096))


# ---------------------------------------------------------------------------
# models and inputs
# ---------------------------------------------------------------------------

def _config(shape, layers, batch, rows, **more):
    c = dict(n_layers=layers, n_kv_heads=0, max_pos=0, n_classes=0, dtype="bf16", norm_eps=1e-5, rope_theta=10000.0,
             hsm_eps=1e-6, kv_block_tokens=16, max_batch=batch, max_pass_tokens=max(rows, batch), max_src=0)
    c.update(SHAPES[shape])
    c.update(more)
    c["n_kv_heads"] = c["n_kv_heads"] or c["n_heads"]
    c.setdefault("hsm_m1", 4 * c["d_model"])
    c.setdefault("hsm_m2", 8 * c["d_model"])
    return SimpleNamespace(**c)


def _weight_shapes(c):
    D, F, dq, dkv = c.d_model, c.d_ffn, c.n_heads * c.head_dim, c.n_kv_heads * c.head_dim
    llama, bert = c.family == "llama", c.family == "bert"
    s = {"tok_emb": (c.vocab, D)}
    if not llama:
        s["pos_emb"] = (c.max_pos, D)
    if bert:
        s.update({"type_emb": (D,), "emb_ln.g": (D,), "emb_ln.b": (D,)})
    for i in range(c.n_layers):
        p = "layers.%d." % i
        s.update({p + "attn_norm.g": (D,), p + "ffn_norm.g": (D,), p + "wq": (dq, D), p + "wk": (dkv, D),
                  p + "wv": (dkv, D), p + "wo": (D, dq)})
        if llama:
            s.update({p + "w_gate": (F, D), p + "w_up": (F, D), p + "w_down": (D, F)})
        else:
            s.update({p + "attn_norm.b": (D,), p + "ffn_norm.b": (D,), p + "bq": (dq,), p + "bk": (dkv,),
                      p + "bv": (dkv,), p + "bo": (D,), p + "w_fc": (F, D), p + "b_fc": (F,), p + "w_proj": (D, F),
                      p + "b_proj": (D,)})
        if c.max_src:
            s.update({p + "cross_norm.g": (D,), p + "cross_norm.b": (D,), p + "cwq": (dq, D), p + "cwk": (dkv, D),
                      p + "cwv": (dkv, D), p + "cwo": (D, dq), p + "cbq": (dq,), p + "cbk": (dkv,), p + "cbv": (dkv,),
                      p + "cbo": (D,)})
    if bert:
        s.update({"pool.w": (D, D), "pool.b": (D,), "cls.w": (c.n_classes, D), "cls.b": (c.n_classes,)})
    else:
        s["final_norm.g"] = (D,)
        if llama:
            s["lm_head"] = (c.vocab, D)
        else:
            s["final_norm.b"] = (D,)
    m1, m2 = c.hsm_m1, c.hsm_m2
    s.update({"hsm.g0": (D,), "hsm.conv_w": (3, 3), "hsm.conv_b": (1,), "hsm.fc1_w": (m1, D), "hsm.fc1_b": (m1,),
              "hsm.fc2_w": (m2, m1), "hsm.fc2_b": (m2,), "hsm.fc3_w": (m1, m2), "hsm.fc3_b": (m1,), "hsm.g1": (m1,),
              "hsm.fc4_w": (D, m1), "hsm.fc4_b": (D,), "hsm.g2": (D,)})
    return s


def _weights(c, seed):
    """A freshly initialised model: N(0, 0.02^2), norm gains 1 and shifts 0, convolution taps N(0, 0.5^2).
    The fp32 model's gains and shifts vary, since nothing rounds there."""
    dt = torch.float32 if c.dtype == "f32" else torch.bfloat16
    g = torch.Generator("cuda").manual_seed(seed)
    vary = 0.1 if c.dtype == "f32" else 0.0
    out = {}
    for name, shape in _weight_shapes(c).items():
        t = torch.empty(shape, dtype=dt, device="cuda")
        if name.endswith(".g") or name in ("hsm.g0", "hsm.g1", "hsm.g2"):
            t.normal_(1.0, vary, generator=g) if vary else t.fill_(1.0)
        elif name.endswith(("norm.b", "ln.b")):
            t.normal_(0.0, vary, generator=g) if vary else t.zero_()
        else:
            t.normal_(0.0, 0.5 if name == "hsm.conv_w" else 0.02, generator=g)
        out[name] = t
    return out


def _tokens(g, c, *shape):
    return torch.randint(0, c.vocab, shape, generator=g, device="cuda", dtype=torch.int32)


def _exits(g, case, *shape):
    if not case["hi"]:
        return None
    return torch.randint(case["lo"], case["hi"] + 1, shape, generator=g, device="cuda", dtype=torch.int32)


#: The fp32 model's threshold, near the median similarity of its random-init states: a part of the tokens leaves at
#: each layer that tests.
DELTA = 0.57


def _inputs(case, seed):
    """Configurations, and the tensors that the calls take."""
    g = torch.Generator("cuda").manual_seed(seed + 1)
    kind = case["kind"]
    s = SimpleNamespace(case=case)
    if kind in ("turn", "encdec"):
        B, P, T = case["batch"], case["prompt"], case["steps"]
        if kind == "turn":
            s.cfg = _config(case["shape"], case["layers"], B, B * P)
        else:
            S = case["source"]
            s.enc_cfg = _config("ofa_enc", case["layers"], B, B * S)
            s.cfg = _config("ofa_dec", case["layers"], B, B * P, max_src=S)
            s.source = _tokens(g, s.enc_cfg, B, S)
            s.source_exits = _exits(g, case, B, S)
        s.prompt, s.exits = _tokens(g, s.cfg, B, P), _exits(g, case, B, P)
        s.step_tokens = [_tokens(g, s.cfg, B) for _ in range(T)]
        s.step_exits = [_exits(g, case, B) for _ in range(T)]
        s.delta = DELTA
    elif kind == "fill":
        n, N = case["tokens"], case["layers"]
        s.cfg = _config(case["shape"], N, 1, 16)
        s.mapped = torch.randn(n, s.cfg.d_model, generator=g, device="cuda").bfloat16()
        s.exits = torch.randint(1, N + 1, (n,), generator=g, device="cuda", dtype=torch.int32)
        s.seq = torch.zeros(n, dtype=torch.int32, device="cuda")
        s.pos = torch.randperm(n, generator=g, device="cuda").to(torch.int32)
    else:
        n = case["rows"]
        s.cfg = _config(case["shape"], case["layers"], 1, 16)
        D = s.cfg.d_model
        rows = lambda std: torch.randn(n, D, generator=g, device="cuda") * std  # noqa: E731
        s.s_prev = rows(1.0)
        s.s_i = s.s_prev + rows(0.3)
        depth = torch.randint(2, 12, (n, 1), generator=g, device="cuda").float()
        s.inertia = (depth - 1) * s.s_prev / s.s_prev.norm(dim=1, keepdim=True) + rows(0.1)
        if s.cfg.family == "bert":
            s.s_final = s.s_i + rows(0.5)
            s.labels = torch.randint(0, s.cfg.n_classes, (-(-n // 128),), generator=g, device="cuda", dtype=torch.int32)
        else:
            s.target = torch.randint(0, s.cfg.vocab, (n,), generator=g, device="cuda", dtype=torch.int32)
    return s


#: A training step's AdamW (within the paper's learning rates and weight decays).
ADAMW = dict(lr=1e-4, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=1e-2)


def prepare(case, seed):
    s = _inputs(case, seed)
    s.model = adept.Model(s.cfg, _weights(s.cfg, seed))
    if case["kind"] == "encdec":
        s.encoder = adept.Model(s.enc_cfg, _weights(s.enc_cfg, seed + 2))
    elif case["kind"] == "fill":
        # every position holds the K/V of a zero state first, so that the whole range can be read back
        n = case["tokens"]
        adept.adept_seq_reserve(s.model.h, [n])
        adept.adept_skip_kv_fill(s.model.h, n, torch.zeros_like(s.mapped), torch.ones_like(s.exits), s.seq, s.pos)
        torch.cuda.synchronize()
    elif case["kind"] == "train":
        adept.adept_hsm_train_init(s.model.h, case["rows"])
        s.loss = torch.zeros(1, device="cuda")
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    kind, m = s.case["kind"], s.model
    if kind in ("turn", "encdec"):
        out = {}
        if kind == "encdec":
            B, S = s.source.shape
            s.encoder.prefill(s.source, s.delta, s.source_exits)
            states = s.encoder.final_states(B * S)
            m.set_cross_source([S] * B, states)
            out["source_states"] = states
        exits, logits, _, sims = m.prefill(s.prompt, s.delta, s.exits)
        out.update(exits=exits, logits=logits, similarities=sims)
        if not s.step_tokens:   # the states are the result; a turn's next steps read them as K/V
            out["states"] = m.final_states(s.prompt.numel())
        out["steps"] = []
        for tokens, forced in zip(s.step_tokens, s.step_exits):
            exits, logits, _, _ = m.decode_step(tokens, s.delta, forced)
            out["steps"].append([exits, logits])
        return out
    if kind == "fill":
        n = s.case["tokens"]
        adept.adept_skip_kv_fill(m.h, n, s.mapped, s.exits, s.seq, s.pos)
        return [list(m.read_kv(layer, 0, 0, n)) for layer in range(2, s.case["layers"] + 1)]
    n = s.case["rows"]
    if s.cfg.family == "bert":
        adept.adept_hsm_train_step_cls(m.h, n, s.s_i, s.s_prev, s.inertia, s.s_final, s.labels, loss_out=s.loss, **ADAMW)
    else:
        adept.adept_hsm_train_step(m.h, n, s.s_i, s.s_prev, s.inertia, s.target, loss_out=s.loss, **ADAMW)
    return {"loss": s.loss, "gradients": [m.hsm_train_read(adept.HSM_GRADS, i) for i in range(len(MAPPER))],
            "parameters": [m.hsm_train_read(adept.HSM_PARAMS, i) for i in range(len(MAPPER))]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _pass_work(c, case, rows, batch, keys, causal_prompt, esz):
    """One early-exit pass of `rows` tokens (`batch` of them give logits; `keys` cached positions of each earlier
    token), with exits uniform on [lo, hi] (the fp32 model: about half of those that may leave at each layer)."""
    N, D, F = c.n_layers, c.d_model, c.d_ffn
    dq, dkv = c.n_heads * c.head_dim, c.n_kv_heads * c.head_dim
    lo, hi = (case["lo"], case["hi"]) if case["hi"] else (2, N)
    n_law = hi - lo + 1
    up = 2 * F if c.family == "llama" else F
    w_layer = D * (dq + 2 * dkv) + dq * D + up * D + F * D
    w_cross = 2 * D * dq if c.max_src else 0
    w_map = 2 * (c.hsm_m1 * D + c.hsm_m1 * c.hsm_m2)
    by = fl = 0.0
    for i in range(1, N + 1):
        stay = 1.0 if i <= lo else max(0.0, (hi - i + 1) / n_law)    # share of tokens that layer i computes
        some = 1.0 - (1.0 - stay) ** rows
        by += some * (w_layer + w_cross) * esz + (1.0 - some) * 2 * dkv * D * esz + 2 * rows * dkv * esz
        fl += 2.0 * rows * (stay * (w_layer + w_cross) + (1.0 - stay) * 2 * D * dkv)
        seen = (keys + 1) / 2.0 if causal_prompt else keys
        fl += 4.0 * rows * stay * dq * (seen + c.max_src)
        if not causal_prompt and c.family != "bert":                 # a generation step reads the cache
            by += rows * stay * keys * 2 * dkv * esz
        by += batch * some * c.max_src * 2 * dkv * esz
        if 2 <= i < N and lo <= i <= hi:
            some = 1.0 - (1.0 - 1.0 / n_law) ** rows if causal_prompt or c.family == "bert" else 1.0 / n_law
            by += some * w_map * esz
            fl += 2.0 * rows / n_law * w_map
    head = D * D if c.family == "bert" else c.vocab * D
    by += head * esz + batch * (c.vocab if c.family != "bert" else c.n_classes) * 4 + rows * (4 + D * esz)
    fl += 2.0 * batch * head
    return by, fl


def work(case):
    kind = case["kind"]
    if kind in ("turn", "encdec"):
        B, P = case["batch"], case["prompt"]
        by = fl = 0.0
        if kind == "turn":
            c = _config(case["shape"], case["layers"], B, B * P)
        else:
            S = case["source"]
            e = _config("ofa_enc", case["layers"], B, B * S)
            c = _config("ofa_dec", case["layers"], B, B * P, max_src=S)
            dkv = c.n_kv_heads * c.head_dim
            by, fl = _pass_work(e, case, B * S, B, S, False, 2)
            by += B * S * e.d_model * 8 + c.n_layers * 2 * dkv * (c.d_model + B * S) * 2
            fl += 2.0 * B * S * c.n_layers * 2 * dkv * c.d_model
        esz = 4 if c.dtype == "f32" else 2
        b, f = _pass_work(c, case, B * P, B, P, c.family != "bert", esz)
        by, fl = by + b, fl + f
        if not case["steps"]:
            by += B * P * c.d_model * 4
        for t in range(case["steps"]):
            b, f = _pass_work(c, case, B, B, P + t + 1, False, esz)
            by, fl = by + b, fl + f
        return {"bytes": by, "flops": fl}
    if kind == "fill":
        n, N = case["tokens"], case["layers"]
        c = _config(case["shape"], N, 1, 16)
        D, kv = c.d_model, 2 * c.n_kv_heads * c.head_dim
        pairs = n * (N - 1) / 2.0                     # exit layers uniform on [1, N]
        by = (N - 1) * kv * D * 2 + n * (D * 2 + 12) + pairs * kv * 2 + 2 * (N - 1) * n * kv * 2
        return {"bytes": by, "flops": 2.0 * pairs * kv * D}
    c = _config(case["shape"], case["layers"], 1, 16)
    n, D = case["rows"], c.d_model
    w = 2 * (c.hsm_m1 * D + c.hsm_m1 * c.hsm_m2)
    labelled = -(-n // 128)
    head = (4.0 * n * c.vocab * D) if c.family != "bert" else 4.0 * labelled * D * D
    by = (D * c.vocab if c.family != "bert" else D * D) * 2 + n * D * (16 if c.family == "bert" else 12)
    # master weights, both moments read and written, the bf16 weights written, gradients and parameters read back
    by += w * (6 * 4 + 2 + 2 * 4)
    return {"bytes": by, "flops": 6.0 * n * w + head}


def tolerance(case):
    """About four times what two implementations of the same precision were seen to differ by: the default kernels
    against the SIMT GEMMs with the mma.sync attention, and against 64 bits."""
    if case["kind"] == "turn" and SHAPES[case["shape"]].get("dtype") == "f32":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}     # 1e-6 against 64 bits
    if case["kind"] == "fill":
        return {"rel": 1e-3, "max": 3e-2}                    # 1.6e-4 and 8e-3: one bf16 rounding of the sum
    if case["kind"] == "train":
        return {"rel": 2e-2, "max": 0.2}                     # up to 5e-3 and 4e-2 (gradients); parameters far less
    if case["kind"] == "turn" and case["shape"].startswith("llama"):
        return {"rel": 3e-2, "max": 0.3, "differ": 0.0}      # 0.7e-2 to 1.6e-2 and 0.08
    return {"rel": 2.4e-2, "max": 0.12, "differ": 0.0}       # 6e-3 and 2.8e-2


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

class _Plain:
    """The early-exit pass of one model in float64: weights as given, nothing rounded."""

    def __init__(self, c, weights):
        self.c, self.w = c, {k: v.double() for k, v in weights.items()}
        self.keys = [None] * c.n_layers
        self.values = [None] * c.n_layers
        self.source = None

    def norm(self, x, name):
        c, w = self.c, self.w
        if c.family == "llama":
            return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + c.norm_eps) * w[name + ".g"]
        return torch.nn.functional.layer_norm(x, x.shape[-1:], w[name + ".g"], w[name + ".b"], c.norm_eps)

    def lin(self, x, w, b=None):
        y = x @ self.w[w].T
        return y + self.w[b] if b in self.w else y

    def heads(self, x, n):
        return x.reshape(*x.shape[:-1], n, self.c.head_dim)

    def turn(self, x, pos):
        """Rotary embedding of x [..., positions, heads, d]: feature i pairs with i + d / 2."""
        if self.c.family != "llama":
            return x
        d = self.c.head_dim
        f = self.c.rope_theta ** (-2.0 * torch.arange(d // 2, dtype=torch.float64, device=x.device) / d)
        a = pos.double()[:, None] * f
        co, si = a.cos()[:, None, :], a.sin()[:, None, :]
        u, v = x[..., :d // 2], x[..., d // 2:]
        return torch.cat([u * co - v * si, v * co + u * si], -1)

    def attend(self, q, k, v, pos, causal):
        c = self.c
        rep = c.n_heads // c.n_kv_heads
        out = []
        for b in range(q.shape[0]):                        # a sequence at a time
            kb = k[b].repeat_interleave(rep, 1)
            vb = v[b].repeat_interleave(rep, 1)
            sc = torch.einsum("nhd,lhd->hnl", q[b], kb) / math.sqrt(c.head_dim)
            if causal:
                hide = torch.arange(kb.shape[0], device=q.device)[None, :] > pos[:, None]
                sc = sc.masked_fill(hide, -math.inf)
            out.append(torch.einsum("hnl,lhd->nhd", sc.softmax(-1), vb).flatten(-2))
        return torch.stack(out)

    def kv(self, i, x, pos):
        c, p = self.c, "layers.%d." % i
        x = x if c.family == "bert" else self.norm(x, p + "attn_norm")
        k = self.turn(self.heads(self.lin(x, p + "wk", p + "bk"), c.n_kv_heads), pos)
        return k, self.heads(self.lin(x, p + "wv", p + "bv"), c.n_kv_heads)

    def layer(self, i, x, pos):
        """Layer i on the states x [B, P, D]; its K/V are in self.keys / self.values."""
        c, p = self.c, "layers.%d." % i
        gelu = torch.nn.functional.gelu
        y = x if c.family == "bert" else self.norm(x, p + "attn_norm")
        q = self.turn(self.heads(self.lin(y, p + "wq", p + "bq"), c.n_heads), pos)
        a = self.attend(q, self.keys[i], self.values[i], pos, c.family != "bert")
        h = x + self.lin(a, p + "wo", p + "bo")
        if c.family == "bert":
            h = self.norm(h, p + "attn_norm")
            return self.norm(h + self.lin(gelu(self.lin(h, p + "w_fc", p + "b_fc")), p + "w_proj", p + "b_proj"),
                             p + "ffn_norm")
        if c.max_src:
            q = self.heads(self.lin(self.norm(h, p + "cross_norm"), p + "cwq", p + "cbq"), c.n_heads)
            k = self.heads(self.lin(self.source, p + "cwk", p + "cbk"), c.n_kv_heads)
            v = self.heads(self.lin(self.source, p + "cwv", p + "cbv"), c.n_kv_heads)
            h = h + self.lin(self.attend(q, k, v, pos, False), p + "cwo", p + "cbo")
        y = self.norm(h, p + "ffn_norm")
        if c.family == "llama":
            f = torch.nn.functional.silu(self.lin(y, p + "w_gate")) * self.lin(y, p + "w_up")
            return h + self.lin(f, p + "w_down")
        return h + self.lin(gelu(self.lin(y, p + "w_fc", p + "b_fc"), approximate="tanh"), p + "w_proj", p + "b_proj")

    def map(self, s, s_prev, inertia):
        return _map(self.w, self.c, s, s_prev, inertia)

    def run(self, tokens, exits, delta, pos):
        """A pass over tokens [B, P] at positions pos [P]: (exit layers, similarities, final states, logits)."""
        c, w, N = self.c, self.w, self.c.n_layers
        x = w["tok_emb"][tokens.long()]
        if c.family != "llama":
            x = x + w["pos_emb"][pos]
        if c.family == "bert":
            x = self.norm(x + w["type_emb"], "emb_ln")
        live = torch.ones(tokens.shape, dtype=torch.bool, device="cuda")
        left = torch.full(tokens.shape, N, dtype=torch.int32, device="cuda")
        sims = torch.full((*tokens.shape, N), math.nan, dtype=torch.float64, device="cuda")
        inertia = torch.zeros_like(x)
        unit = lambda t: t / t.norm(dim=-1, keepdim=True)  # noqa: E731
        for i in range(N):
            # an exited token's x is its mapped state: its K/V of this layer come from it
            k, v = self.kv(i, x, pos)
            if pos[0] == 0:
                self.keys[i], self.values[i] = k, v
            else:
                self.keys[i], self.values[i] = torch.cat([self.keys[i], k], 1), torch.cat([self.values[i], v], 1)
            if not live.any():
                continue
            y = torch.where(live[..., None], self.layer(i, x, pos), x)
            if 1 <= i < N - 1:
                cos = (unit(y) * unit(inertia)).sum(-1)
                sims[..., i] = torch.where(live, cos, sims[..., i])
                go = live & (cos >= delta if exits is None else exits == i + 1)
                if go.any():
                    mapped = self.map(y[go], x[go], inertia[go])
                    y = y.index_put((go,), mapped)
                    left[go] = i + 1
                    live = live & ~go
            inertia = torch.where(live[..., None], inertia + unit(y), inertia)
            x = y
        if c.family == "bert":
            logits = self.lin(torch.tanh(self.lin(x[:, 0], "pool.w", "pool.b")), "cls.w", "cls.b")
        else:
            logits = self.norm(x[:, -1], "final_norm") @ w["lm_head" if c.family == "llama" else "tok_emb"].T
        return left.reshape(-1), sims.reshape(-1, N), x.reshape(-1, c.d_model), logits


def _map(w, c, s, s_prev, inertia):
    """The hidden-state mapper on rows [n, D]."""
    rms = lambda t, g: t * torch.rsqrt(t.square().mean(-1, keepdim=True) + c.hsm_eps) * w[g]  # noqa: E731
    gelu = torch.nn.functional.gelu
    three = torch.stack([rms(s, "hsm.g0"), rms(s_prev, "hsm.g0"), rms(inertia, "hsm.g0")], 1)
    pad = torch.nn.functional.pad(three, (1, 1))
    D = s.shape[-1]
    c0 = w["hsm.conv_b"] + sum(w["hsm.conv_w"][a, u] * pad[:, a, u:u + D] for a in range(3) for u in range(3))
    h1 = gelu(c0 @ w["hsm.fc1_w"].T + w["hsm.fc1_b"])
    h2 = gelu(h1 @ w["hsm.fc2_w"].T + w["hsm.fc2_b"])
    h4 = rms(h2 @ w["hsm.fc3_w"].T + w["hsm.fc3_b"], "hsm.g1") + h1
    return rms(h4 @ w["hsm.fc4_w"].T + w["hsm.fc4_b"], "hsm.g2") + c0


def _exact_train(s, weights):
    c, n = s.cfg, s.case["rows"]
    w = {k: v.double() for k, v in weights.items()}
    for k in MAPPER:
        w[k].requires_grad_(True)
    st = _map(w, c, s.s_i.double(), s.s_prev.double(), s.inertia.double())
    F = torch.nn.functional
    if c.family == "bert":
        loss = (1.0 - F.cosine_similarity(st, s.s_final.double(), dim=-1)).mean()
        r = len(s.labels)
        pooled = torch.tanh(st[:r] @ w["pool.w"].T + w["pool.b"])
        loss = loss + F.cross_entropy(pooled @ w["cls.w"].T + w["cls.b"], s.labels.long())
    else:
        y = F.layer_norm(st, (c.d_model,), w["final_norm.g"], w["final_norm.b"], c.norm_eps)
        loss = F.cross_entropy(y @ w["tok_emb"].T, s.target.long())
    grads = torch.autograd.grad(loss, [w[k] for k in MAPPER])
    a = ADAMW
    new = []
    for k, g in zip(MAPPER, grads):                          # AdamW's first step from zero moments
        t = w[k].detach()
        new.append((t - a["lr"] * a["weight_decay"] * t - a["lr"] * g / (g.abs() + a["eps"])).reshape(-1))
    return {"loss": loss.detach().reshape(1), "gradients": [g.reshape(-1) for g in grads], "parameters": new}


@torch.no_grad()
def exact(case, seed):
    s = _inputs(case, seed)
    weights = _weights(s.cfg, seed)
    if case["kind"] == "train":
        with torch.enable_grad():
            return _exact_train(s, weights)
    m = _Plain(s.cfg, weights)
    if case["kind"] == "fill":
        n, out = case["tokens"], []
        x = torch.empty(n, s.cfg.d_model, dtype=torch.float64, device="cuda")
        x[s.pos.long()] = s.mapped.double()
        left = torch.empty_like(s.exits)
        left[s.pos.long()] = s.exits
        pos = torch.arange(n, device="cuda")
        for i in range(1, case["layers"]):
            filled = (left <= i)[:, None, None]
            out.append([t[0] * filled for t in m.kv(i, x[None], pos)])
        return out
    out = {}
    P = case["prompt"]
    if case["kind"] == "encdec":
        S = case["source"]
        e = _Plain(s.enc_cfg, _weights(s.enc_cfg, seed + 2))
        states = e.run(s.source, s.source_exits, s.delta, torch.arange(S, device="cuda"))[2]
        m.source = states.reshape(case["batch"], S, -1)
        out["source_states"] = states
    exits, sims, states, logits = m.run(s.prompt, s.exits, s.delta, torch.arange(P, device="cuda"))
    out.update(exits=exits, logits=logits, similarities=sims)
    if not s.step_tokens:
        out["states"] = states
    out["steps"] = []
    for t, (tokens, forced) in enumerate(zip(s.step_tokens, s.step_exits)):
        exits, _, _, logits = m.run(tokens[:, None], None if forced is None else forced[:, None], s.delta,
                                    torch.arange(P + t, P + t + 1, device="cuda"))
        out["steps"].append([exits, logits])
    return out
