"""The work a serving program has this library do, as cases that can be timed and compared.

One request's life on the affix-cache path: the probe with its selection (once per request), refresh passes over the
anchors and the request's own rows, decode passes over the block being denoised, and the single-layer step that chains
scoring, selection, recomputation and scatter.  Shapes are those of the configurations and tests of this repository
(LLaDA-8B-, Dream-7B-shaped and tiny layers).  Every layer of a model is the same work, so the multi-layer calls run a
few layers, each with weights and caches of its own (more than the L2 cache holds), followed by the whole LM head.

Inputs are drawn on the device from the seed.  Two things make them behave as trained models do where random ones would
not: query and key projections are correlated and the masked rows share a direction with the rows that end up as
anchors (attention to the affix concentrates on few tokens, so the selection is not decided by the last bit), and the
LM head's rows of the predicted tokens lie along the hidden states (predictions are confident).
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import torch

from paper_2608_26140_b200 import binding as ab
from paper_2608_26140_b200 import workloads as wl

DEV = "cuda:0"
MODELS = {"llada-8b": (wl.LLADA_8B, 126464), "dream-7b": (wl.DREAM_7B, 152064), "tiny": (wl.TINY, 2048),
          "tiny-gqa": (wl.TINY_GQA, 2048)}
LAYER_KINDS = ("layer_step", "layer_step_host")


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _case(kind, model, batch, pre, affix, post, gen, masked, ratio, extra, layers=1, shared=False, name=None):
    """The context is [pre request rows][affix][post request rows][gen rows]; the first `masked` generation rows are
    the masked ones.  extra: which rows are recomputed beside the anchors ("none", "masked", "all" non-affix rows)."""
    c = dict(kind=kind, model=model, batch=batch, pre=pre, affix=affix, post=post, gen=gen, masked=masked, ratio=ratio,
             extra=extra, layers=layers, shared=shared)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # smallest call: the tiny layer, one request; launches and latency
        _case("layer_step", "tiny", 1, 0, 128, 64, 64, 32, 0.2, "masked", name="layer-step-tiny"),
        # one request, 512-token prefix, anchors only: the layer-step the benchmark leads with; weight streaming
        _case("layer_step", "llada-8b", 1, 0, 512, 256, 256, 32, 0.2, "none", name="layer-step-b1"),
        # the same from host buffers: a caller whose hidden states live in pinned host memory
        _case("layer_step_host", "llada-8b", 1, 0, 512, 256, 256, 32, 0.2, "none", name="layer-step-host-b1"),
        # the same with every request row recomputed, as the method is published; a few hundred rows
        _case("layer_step", "llada-8b", 1, 0, 512, 256, 256, 32, 0.2, "all", name="layer-step-b1-all-rows"),
        # one request with a long affix in the middle: scoring, selection and attention over 8192 keys
        _case("layer_step", "llada-8b", 1, 32, 8192, 32, 32, 32, 0.2, "none", name="layer-step-long-affix"),
        # many requests with a short affix: thousands of rows over few keys each
        _case("layer_step", "llada-8b", 64, 0, 512, 64, 32, 32, 0.2, "none", name="layer-step-b64"),
        # grouped heads and biases, sizes that divide nothing
        _case("layer_step", "dream-7b", 5, 77, 1337, 41, 67, 29, 0.13, "masked", name="layer-step-ragged-gqa"),
        # one denoising step that refreshes anchors and all request rows of a full batch
        _case("refresh", "llada-8b", 16, 0, 2048, 256, 256, 32, 0.2, "all", layers=2, name="refresh-b16"),
        # decode pass of a single request: 32 block rows through the layers and the LM head
        _case("decode", "llada-8b", 1, 0, 512, 256, 256, 32, 0.2, "masked", layers=4, name="decode-b1"),
        # decode pass of a full batch over one shared copy of the affix cache and private slots
        _case("decode", "llada-8b", 16, 0, 2048, 256, 256, 32, 0.2, "masked", layers=4, shared=True, name="decode-shared-b16"),
        # probe and selection of a full batch, affix in the middle, grouped heads
        _case("probe", "dream-7b", 32, 128, 1024, 256, 256, 256, 0.2, "all", layers=2, name="probe-b32-gqa"),
        # the other selector: K/V deviation of every affix token, then the same selection
        _case("kv_deviation", "llada-8b", 8, 0, 2048, 64, 32, 32, 0.2, "none", name="kv-deviation-b8"),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    most = max(_seconds(c) for c in listed())
    while True:
        kind = rng.choice(("layer_step", "layer_step", "layer_step_host", "refresh", "decode", "decode", "probe", "kv_deviation"))
        model = rng.choice(("llada-8b", "llada-8b", "dream-7b", "dream-7b", "tiny", "tiny-gqa"))
        tiny = model.startswith("tiny")
        most_batch = 4 if kind == "layer_step_host" else 8 if tiny else 64
        batch, affix = log_int(1, most_batch), log_int(64, 256 if tiny else 8192)
        gen = rng.choice((32, 64, 128, 256)) if rng.random() < 0.5 else log_int(32, 256)
        masked = min(gen, 32) if rng.random() < 0.5 else rng.randint(8, min(gen, 64))
        pre, post = rng.choice((0, 0, log_int(1, 256))), log_int(8, 256)
        ratio = rng.choice((0.05, 0.1, 0.2, 0.2, 0.35, 0.5, round(rng.uniform(0.05, 0.5), 3)))
        extra = {"refresh": "all", "probe": "all", "decode": "masked", "kv_deviation": "none", "layer_step_host": "none",
                 "layer_step": rng.choice(("none", "masked", "all"))}[kind]
        layers = rng.randint(2, 4) if kind in ("refresh", "decode", "probe") else 1
        if kind == "probe":
            masked = gen
        shared = kind in ("refresh", "decode") and rng.random() < 0.5
        c = _case(kind, model, batch, pre, affix, post, gen, masked, ratio, extra, layers, shared)
        rows = batch * (pre + post + gen + int(ratio * affix))
        if _seconds(c) < 0.7 * most and rows <= 16384 and _cache_bytes(c) < 10e9:
            return c


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def _sizes(case):
    s, vocab = MODELS[case["model"]]
    T = case["pre"] + case["affix"] + case["post"] + case["gen"]
    k = max(0, min(case["affix"], math.ceil(case["ratio"] * case["affix"] - 1e-9)))
    extra = {"none": 0, "masked": case["masked"], "all": T - case["affix"]}[case["extra"]]
    return s, vocab, T, k, extra


def _cache_bytes(case):
    s, _, T, _, _ = _sizes(case)
    return case["layers"] * case["batch"] * T * 2 * s.kv_dim * 2


def work(case):
    s, vocab, T, k, e = _sizes(case)
    B, L, m, n_layers, kind = case["batch"], case["affix"], case["masked"], case["layers"], case["kind"]
    D, F, kvb = s.hidden, s.ffn, 2 * s.kv_dim * 2            # kvb: K and V bytes of one position
    select = 8 * B * L + 4 * B * k
    if kind == "kv_deviation":
        return {"bytes": 2 * B * L * kvb + select, "flops": 6 * B * L * s.kv_dim}
    score = kind in LAYER_KINDS
    rows = B * {"decode": e, "probe": e}.get(kind, k + e)
    # keys and values read: every request's own context, or one shared affix and the private rows
    kept = B * (T - L + k) + L if case["shared"] else B * T
    params = D * s.q_dim + 2 * D * s.kv_dim + s.q_dim * D + 3 * D * F
    q_rows = B * m if score else 0                             # masked rows' queries, the step's own scoring
    n_bytes = n_layers * (2 * params + kept * kvb + rows * kvb) + (2 * rows + q_rows) * D * 2
    n_flops = n_layers * (2 * rows * params + 4 * rows * T * s.q_dim) + 2 * q_rows * D * s.q_dim
    if score or kind == "probe":
        n_bytes += select
        n_flops += n_layers * 2 * B * m * L * s.q_dim
    if kind in ("refresh", "decode"):
        n_bytes += 2 * vocab * D
        n_flops += 2 * B * m * D * vocab
    return {"bytes": n_bytes, "flops": n_flops}


def _seconds(case):
    w = work(case)
    return max(w["bytes"] / 6e12, w["flops"] / 1.4e15)


def tolerance(case):
    if case["kind"] == "kv_deviation":
        return {"rel": 4e-6}                                   # fp32 sums of thousands of squares; the selection is exact
    # bf16 storage between the stages: a rounding flip moves an element by 2^-8, and the layers add up.  The library's
    # mma.sync kernels and one-SM projections against its tcgen05 and two-SM ones: 3e-3 after one layer, 4.5e-3 after
    # two, 7e-3 after four, single elements 0.04; four times that
    return {"rel": min(0.03, 6e-3 * (1 + case["layers"])), "max": 0.15, "differ": 0.005}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _weights(s, T, randn):
    """One layer's weights at the scale of unit-variance activations.  In the rotary pairs too slow to turn within the
    context, queries correlate with the keys they read; a layer's update is small against the residual stream."""
    std = 1.28 / math.sqrt(s.hidden)
    half = s.head_dim // 2
    slow = (s.rope_theta ** (-torch.arange(half, device=DEV) / half) * T < 1.5).repeat(2).to(torch.bfloat16).view(-1, 1)
    wk = randn((s.n_kv_heads, s.head_dim, s.hidden), std)
    wq = randn((s.n_kv_heads, s.n_heads // s.n_kv_heads, s.head_dim, s.hidden), std)
    wq = wq.mul_(1 - 0.7 * slow).add_((wk * slow).unsqueeze(1), alpha=0.95)
    w = dict(attn_norm_g=randn((s.hidden,), 0.05).add_(1), wq=wq.view(s.q_dim, s.hidden), wk=wk.view(s.kv_dim, s.hidden),
             wv=randn((s.kv_dim, s.hidden), std), wo=randn((s.hidden, s.q_dim), 0.3 * std),
             mlp_norm_g=randn((s.hidden,), 0.05).add_(1), w_gate=randn((s.ffn, s.hidden), std),
             w_up=randn((s.ffn, s.hidden), std), w_down=randn((s.hidden, s.ffn), 0.3 * std))
    if s.qkv_bias:
        w.update(bq=randn((s.q_dim,), 0.02), bk=randn((s.kv_dim,), 0.02), bv=randn((s.kv_dim,), 0.02))
    return w


def _affix_cache(s, w, x, start, cos, sin):
    """K (after the rotary embedding) and V of the affix rows x [L, D] under these weights, as a cache holds them."""
    xn = torch.nn.functional.rms_norm(x.float(), (s.hidden,), w["attn_norm_g"].float(), s.rms_eps).to(torch.bfloat16)
    k, v = xn @ w["wk"].T, xn @ w["wv"].T
    if s.qkv_bias:
        k, v = k + w["bk"], v + w["bv"]
    L = x.shape[0]
    lo, hi = k.float().view(L, s.n_kv_heads, 2, s.head_dim // 2).unbind(2)
    c, n = cos[start:start + L, None], sin[start:start + L, None]
    k = torch.cat((lo * c - hi * n, hi * c + lo * n), -1).to(torch.bfloat16)
    return k, v.view(L, s.n_kv_heads, s.head_dim)


def prepare(case, seed):
    s, vocab, T, k, _ = _sizes(case)
    B, L, l, m, kind = case["batch"], case["affix"], case["pre"], case["masked"], case["kind"]
    gen = torch.Generator(device=DEV).manual_seed(int(seed))

    def randn(shape, std=1.0):
        t = torch.randn(shape, generator=gen, device=DEV, dtype=torch.bfloat16)
        return t.mul_(std) if std != 1.0 else t

    def positions(*spans):
        p = torch.cat([torch.arange(a, b, dtype=torch.int32, device=DEV) for a, b in spans])
        return p.expand(B, -1).contiguous()

    st = SimpleNamespace(case=case, k=k)
    lay = wl.make_layout(B, l, L, case["post"], case["gen"], m, case["extra"])
    masked = positions((lay.ctx_len - case["gen"], lay.ctx_len - case["gen"] + m))
    extra = {"none": None, "masked": masked, "all": positions((0, l), (l + L, T))}[case["extra"]]
    n = lay.n_extra if kind in ("decode", "probe") else k + lay.n_extra
    cos_h, sin_h = wl.rope_table(T, s.head_dim, s.rope_theta)
    cos, sin = torch.from_numpy(cos_h).to(DEV), torch.from_numpy(sin_h).to(DEV)
    st.keep = [masked, extra, cos, sin]

    st.anchors = torch.randperm(L, generator=gen, device=DEV)[:k].sort().values.to(torch.int32).expand(B, -1).contiguous()
    # hidden states: the affix text is the same for every request, each row carries its context's share; where anchors
    # are selected, the masked rows and the rows that will be the anchors have one direction in common
    st.x = randn((B, T, s.hidden))
    affix = randn((L, s.hidden))
    at, mp = st.anchors[0].long(), masked[0].long()
    if kind in LAYER_KINDS + ("probe",):
        common = randn((s.hidden,), math.sqrt(0.9))
        affix[at] = affix[at] * math.sqrt(0.1) + common
        st.x[:, mp] = st.x[:, mp] * math.sqrt(0.1) + common
    st.x[:, l:l + L] = affix + 0.2 * st.x[:, l:l + L]

    n_caches = 1 if case["shared"] else B
    kv_std = 1.28
    st.w = [_weights(s, T, randn) for _ in range(case["layers"])]
    st.lw = [ab.Context.weights(w) for w in st.w]
    st.caches = []
    for w in st.w:
        ck, cv = (randn((n_caches, T, s.n_kv_heads, s.head_dim), kv_std) for _ in range(2))
        ck[:, l:l + L], cv[:, l:l + L] = _affix_cache(s, w, affix, l, cos, sin)
        st.caches.append((ck, cv))
    st.kvs = [ab.Context.kv(*c) for c in st.caches]
    if case["shared"]:
        for kv in st.kvs:
            kv.batch_stride = 0
    st.req = ab.Context.request(B, T, l, L, masked, extra, cos, sin)
    st.scores = torch.zeros((B, L), dtype=torch.float32, device=DEV)
    st.picked = torch.zeros((B, k), dtype=torch.int32, device=DEV)
    st.y, st.y2 = (torch.zeros((B, max(n, 1), s.hidden), dtype=torch.bfloat16, device=DEV) for _ in range(2))

    blk = vocab_max = 0
    if kind in ("refresh", "decode"):
        blk, vocab_max = m, vocab
        st.norm_g, st.w_lm = randn((s.hidden,), 0.05).add_(1), randn((vocab, s.hidden), 1.28 / math.sqrt(s.hidden))
        said = torch.randperm(vocab, generator=gen, device=DEV)[:B * m]
        st.w_lm[said] += st.x[:, mp].reshape(B * m, s.hidden) * (0.4 / math.sqrt(s.hidden))
        st.token, st.commit = (torch.zeros((B, m), dtype=torch.int32, device=DEV) for _ in range(2))
        st.confidence = torch.zeros((B, m), dtype=torch.float32, device=DEV)
        # compact rows of the block: behind the anchors and the request rows in front of them, or the rows themselves
        first = 0 if kind == "decode" else k + l + case["post"]
        st.block = positions((first, first + m))
    if kind == "decode" and case["shared"]:
        # the private slots a refresh pass over the anchors and all request rows has left
        own = positions((0, l), (l + L, T))
        st.keep.append(own)
        st.req_slots = ab.Context.request(B, T, l, L, masked, own, cos, sin)
        st.slot_rows = positions((k + l + case["post"], k + l + case["post"] + m))
    if case["shared"]:
        slots = k + (T - L)
        st.k_slots = [randn((B, slots, s.n_kv_heads, s.head_dim), kv_std) for _ in st.w]
        st.v_slots = [randn((B, slots, s.n_kv_heads, s.head_dim), kv_std) for _ in st.w]
    if kind == "kv_deviation":
        # the full-prompt cache: the affix-only one plus what the context changes, most at the anchors
        size = torch.full((L, 1, 1), 0.05, device=DEV, dtype=torch.bfloat16)
        size[at] = 0.3
        st.full = [t.clone() for t in st.caches[0]]
        for t in st.full:
            t[:, l:l + L] += randn((B, L, s.n_kv_heads, s.head_dim)) * size
        st.kv_full = ab.Context.kv(*st.full)
    if kind == "layer_step_host":
        st.x = st.x.cpu().pin_memory()
        st.scores, st.picked, st.y = (t.cpu().pin_memory() for t in (st.scores, st.picked, st.y))
    rows = k + (T - L) if case["shared"] else max(n, 1)
    st.ctx = ab.Context.for_shape(s, B, T, L, rows, m, DEV, max_vocab=vocab_max, max_block=blk)
    return st


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def run(st):
    c, ctx = st.case, st.ctx
    kind, ratio = c["kind"], c["ratio"]
    if kind == "layer_step":
        ctx.layer_step(st.lw[0], st.req, st.kvs[0], st.x, 0, ratio, ab.F_SCORE | ab.F_SELECT, st.scores, st.picked, st.y)
        return st.scores, st.picked, st.y, st.caches
    if kind == "layer_step_host":
        ctx.layer_step_host(st.lw[0], st.req, st.kvs[0], st.x, ratio, 0, st.scores, st.picked, st.y)
        return st.scores, st.picked, st.y, st.caches
    if kind == "probe":
        ctx.probe_select(st.lw, st.kvs, st.req, st.x, ratio, 0, st.y, st.y2, st.scores, st.picked)
        return st.scores, st.picked, st.y2 if c["layers"] % 2 == 0 else st.y, st.caches
    if kind == "kv_deviation":
        ctx.score_kv_deviation(st.req, st.kvs[0], st.kv_full, st.scores)
        ctx.select_topk(st.scores, c["batch"], c["affix"], st.k, st.picked)
        return st.scores, st.picked
    head = (st.block, c["masked"], st.norm_g, st.w_lm, st.w_lm.shape[0], 0.9, st.token, st.confidence, st.commit)
    last = st.y2 if c["layers"] % 2 == 0 else st.y
    if c["shared"]:
        if kind == "refresh":
            ctx.denoise_step_shared(st.lw, st.kvs, st.req, st.x, st.anchors, st.k, st.k_slots, st.v_slots, st.y, st.y2, *head)
        else:
            ctx.decode_step_shared(st.lw, st.kvs, st.req, st.req_slots, st.x, st.anchors, st.k, st.slot_rows, st.k_slots,
                                   st.v_slots, st.y, st.y2, *head)
        return last, st.k_slots, st.v_slots, st.token, st.confidence, st.commit
    if kind == "refresh":
        ctx.denoise_step(st.lw, st.kvs, st.req, st.x, st.anchors, st.k, st.y, st.y2, *head)
    else:
        ctx.denoise_step(st.lw, st.kvs, st.req, st.x, None, 0, st.y, st.y2, *head)
    return last, st.caches, st.token, st.confidence, st.commit
