"""Names of the kernels that a call launches, by layer shape and sizes.

A process of its own: the profiler's clock, once started, drifts against the device's, and a later profile of the same process can
lose its kernels (their times lie outside its window)."""
import json
import subprocess
import sys
import time


def launched_kernels(cases, call="rows"):
    """cases: list of (LayerShape, *sizes), as the function `call` of this file takes them -> list of texts, the names of the kernels
    of each."""
    asked = json.dumps([call, [[list(vars(s).values()), *sizes] for s, *sizes in cases]])
    r = subprocess.run([sys.executable, __file__], input=asked, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.splitlines()[-1])


def zeros(*shape):
    return torch.zeros(shape, dtype=torch.bfloat16, device="cuda:0")


def weights(s):
    D, Q, KV, F = s.hidden, s.q_dim, s.kv_dim, s.ffn
    w = dict(attn_norm_g=zeros(D), wq=zeros(Q, D), wk=zeros(KV, D), wv=zeros(KV, D), wo=zeros(D, Q), mlp_norm_g=zeros(D),
             w_gate=zeros(F, D), w_up=zeros(F, D), w_down=zeros(D, F))
    if s.qkv_bias:
        w.update(bq=zeros(Q), bk=zeros(KV), bv=zeros(KV))
    return w


def on_device(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def rope(s, T):
    return [on_device(t) for t in wl.rope_table(T, s.head_dim, s.rope_theta)]


def names(ctx, call):
    for _ in range(3):                       # again if the profile has lost some
        before = ctx.launch_count()
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            time.sleep(0.05)
            call()
            torch.cuda.synchronize()
            time.sleep(0.05)
        assert ctx.poll_status() == 0
        found = [e for e in prof.key_averages() if "kernel" in e.key]
        if sum(e.count for e in found) >= ctx.launch_count() - before:
            break
    return " ".join(e.key for e in found)


def rows(shape, n):
    """recompute_anchors of n anchors of one request"""
    L = n + 8
    lay = wl.make_layout(1, 0, L, 8, 8, 8, "none")
    w, (cos, sin), masked = weights(shape), rope(shape, lay.ctx_len), on_device(lay.masked_pos)
    cache = [zeros(1, lay.ctx_len, shape.n_kv_heads, shape.head_dim) for _ in range(2)]
    new = [zeros(1, n, shape.n_kv_heads, shape.head_dim) for _ in range(2)]
    x, y, anchors = zeros(1, lay.ctx_len, shape.hidden), zeros(1, n, shape.hidden), torch.arange(n, dtype=torch.int32, device="cuda:0")[None].contiguous()
    ctx = ab.Context.for_shape(shape, 1, lay.ctx_len, L, n, 8, "cuda:0")
    req = ab.Context.request(1, lay.ctx_len, 0, L, masked, None, cos, sin)
    return names(ctx, lambda: ctx.recompute_anchors(ab.Context.weights(w), req, ab.Context.kv(*cache), x, 0, anchors, n, *new, y))


def shared_decode(shape, B, pre, L, post, n, K):
    """recompute_rows_shared of n block rows of each of B requests, K anchors each, the affix behind `pre` and in front of `post` rows"""
    lay = wl.make_layout(B, pre, L, post, n, n, "all")
    T, w, (cos, sin), block = lay.ctx_len, weights(shape), rope(shape, lay.ctx_len), on_device(lay.masked_pos)
    cache = [zeros(1, T, shape.n_kv_heads, shape.head_dim) for _ in range(2)]
    slots = [zeros(B, K + lay.n_extra, shape.n_kv_heads, shape.head_dim) for _ in range(2)]
    x, y = zeros(B, T, shape.hidden), zeros(B, n, shape.hidden)
    anchors = torch.arange(K, dtype=torch.int32, device="cuda:0").expand(B, -1).contiguous()
    slot_rows = (K + lay.n_extra - n + torch.arange(n, dtype=torch.int32, device="cuda:0")).expand(B, -1).contiguous()
    extra = on_device(lay.extra_rows)
    ctx = ab.Context.for_shape(shape, B, T, L, K + lay.n_extra, n, "cuda:0")
    req, owned = ab.Context.request(B, T, pre, L, block, block, cos, sin), ab.Context.request(B, T, pre, L, block, extra, cos, sin)
    kv = ab.KV(cache[0].data_ptr(), cache[1].data_ptr(), 0, T)
    return names(ctx, lambda: ctx.recompute_rows_shared(ab.Context.weights(w), req, owned, kv, x, 0, anchors, K, slot_rows, *slots, y))


def scoring(shape, B, L, m, shared, norm_full):
    """score_anchors of m masked rows over L affix keys, 7 rows in front of them"""
    lay = wl.make_layout(B, 7, L, 20, max(m, 8), m)
    cache, q = zeros(1 if shared else B, lay.ctx_len, shape.n_kv_heads, shape.head_dim), zeros(B, m, shape.n_heads, shape.head_dim)
    masked, scores = on_device(lay.masked_pos), torch.zeros((B, L), device="cuda:0")
    ctx = ab.Context.for_shape(shape, B, lay.ctx_len, L, 1, m, "cuda:0")
    req = ab.Context.request(B, lay.ctx_len, 7, L, masked, None, None, None)
    kv = ab.KV(cache.data_ptr(), cache.data_ptr(), 0, lay.ctx_len) if shared else ab.Context.kv(cache, cache)
    return names(ctx, lambda: ctx.score_anchors(req, q, kv, scores, accumulate=False, norm_full=norm_full))


if __name__ == "__main__":
    import os
    import numpy as np
    import torch
    sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    from paper_2608_26140_b200 import binding as ab
    from paper_2608_26140_b200 import workloads as wl
    which, cases = json.load(sys.stdin)
    print(json.dumps([globals()[which](wl.LayerShape(*fields), *sizes) for fields, *sizes in cases]))
