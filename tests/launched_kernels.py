"""Names of the kernels that recompute_anchors launches, by layer shape and row count.

A process of its own: the profiler's clock, once started, drifts against the device's, and a later profile of the same process can
lose its kernels (their times lie outside its window)."""
import json
import subprocess
import sys
import time


def launched_kernels(cases):
    """cases: list of (LayerShape, rows) -> list of texts, the names of the kernels of each."""
    asked = json.dumps([[list(vars(s).values()), rows] for s, rows in cases])
    r = subprocess.run([sys.executable, __file__], input=asked, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.splitlines()[-1])


def names(shape, rows):
    import torch
    from paper_2608_26140_b200 import binding as ab
    from paper_2608_26140_b200 import workloads as wl
    dev, L = "cuda:0", rows + 8
    lay = wl.make_layout(1, 0, L, 8, 8, 8, "none")
    zeros = lambda *s: torch.zeros(s, dtype=torch.bfloat16, device=dev)
    D, Q, KV, F = shape.hidden, shape.q_dim, shape.kv_dim, shape.ffn
    w = dict(attn_norm_g=zeros(D), wq=zeros(Q, D), wk=zeros(KV, D), wv=zeros(KV, D), wo=zeros(D, Q), mlp_norm_g=zeros(D),
             w_gate=zeros(F, D), w_up=zeros(F, D), w_down=zeros(D, F))
    if shape.qkv_bias:
        w.update(bq=zeros(Q), bk=zeros(KV), bv=zeros(KV))
    cos, sin = (torch.from_numpy(t).to(dev) for t in wl.rope_table(lay.ctx_len, shape.head_dim, shape.rope_theta))
    masked = torch.from_numpy(lay.masked_pos.copy()).to(dev)
    cache = [zeros(1, lay.ctx_len, shape.n_kv_heads, shape.head_dim) for _ in range(2)]
    new = [zeros(1, rows, shape.n_kv_heads, shape.head_dim) for _ in range(2)]
    x, y, anchors = zeros(1, lay.ctx_len, D), zeros(1, rows, D), torch.arange(rows, dtype=torch.int32, device=dev)[None].contiguous()
    ctx = ab.Context.for_shape(shape, 1, lay.ctx_len, L, rows, 8, dev)
    req = ab.Context.request(1, lay.ctx_len, 0, L, masked, None, cos, sin)
    for _ in range(3):                       # again if the profile has lost some
        before = ctx.launch_count()
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            time.sleep(0.05)
            ctx.recompute_anchors(ab.Context.weights(w), req, ab.Context.kv(*cache), x, 0, anchors, rows, *new, y)
            torch.cuda.synchronize()
            time.sleep(0.05)
        assert ctx.poll_status() == 0
        found = [e for e in prof.key_averages() if "kernel" in e.key]
        if sum(e.count for e in found) >= ctx.launch_count() - before:
            break
    return " ".join(e.key for e in found)


if __name__ == "__main__":
    import os
    sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    from paper_2608_26140_b200.workloads import LayerShape
    print(json.dumps([names(LayerShape(*fields), rows) for fields, rows in json.load(sys.stdin)]))
