"""Sizes at the edges of the kernels' dispatch rules and tiles, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import acache_oracle as orc
from paper_2608_26140_b200 import binding as ab
from paper_2608_26140_b200 import workloads as wl

from helpers import DEV, DeviceCase, assert_close_bf16, cached_weights, oracle_step
from launched_kernels import launched_kernels
from test_gpu_parity import MID128, check_against_oracle, run_layer_step, run_split_calls
from test_gpu_predict_commit import test_predict_commit as check_predict_commit

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,B,n_blk", [
    (1280, 4, 32),        # 128 rows: the last size of the one-SM kernel
    (1280, 3, 43),        # 129 rows, few tiles: one SM, the second row tile nearly empty
    (2048, 19, 31),       # 589 rows, three row pairs, few tiles: one SM
    (2048, 29, 31),       # 899 rows, four row pairs: two SMs, tiles cut between the clusters
    (2688, 3, 43),        # an odd number of 128-wide vocabulary units: one SM
    (65536, 5, 29),       # whole tiles, 145 rows
    (16384, 19, 31),      # whole tiles, 589 rows: three row pairs, the last one without a second row tile
])
def test_lm_head_tiles(V, B, n_blk):
    check_predict_commit(wl.TINY, V, B, 64, n_blk)


def test_lm_head_cut_tiles():     # K = 2048: ten pair tiles of 129 rows on one SM, 32 of 780 cut between the clusters
    shape = wl.LayerShape(2048, 2, 1, 128, 256, 1e-5, False, 5e5, "lm-head-cut")
    check_predict_commit(shape, 2560, 3, 64, 43)
    check_predict_commit(shape, 2048, 13, 64, 60)


@pytest.mark.parametrize("T", [51200, 51201])     # the last context whose position map fits shared memory, the first past it
def test_position_maps_of_long_contexts(T):
    # slot map of the split call (with two rows naming one position), lookup of the masked rows in a compact input
    lay = wl.make_layout(1, 5, T - 5 - 40, 8, 32, 32, "masked")
    lay.extra_rows = lay.extra_rows.copy()
    lay.extra_rows[0, 3] = lay.extra_rows[0, 20]
    case = wl.make_case(wl.TINY, lay, 0.0, cfg_id=71)
    dc = DeviceCase(case, max_rows=64)
    K = 7
    anchors = np.sort(np.random.default_rng(T).choice(lay.affix_len, K, replace=False)).astype(np.int32)[None]
    k_new, v_new, y = run_split_calls(dc, torch.from_numpy(anchors).to(DEV), K)
    assert dc.ctx.poll_status() == 0
    ref = oracle_step(case, 0, anchor_idx=anchors[0])
    assert_close_bf16(ab.to_host_bits(y[0]), ref["y"], "y")

    lay.extra_rows[0] = lay.masked_pos[0]
    dc = DeviceCase(case, max_rows=64)
    compact = dc.x[:, torch.from_numpy(lay.extra_rows[0]).long().to(DEV)].contiguous()
    scores = torch.zeros((2, lay.affix_len), dtype=torch.float32, device=DEV)
    y = torch.zeros((1, lay.n_extra, case.shape.hidden), dtype=torch.bfloat16, device=DEV)
    for i, (x, is_compact) in enumerate(((dc.x, 0), (compact, 1))):
        dc.ctx.layer_step(dc.lw, dc.req, dc.kv(), x, is_compact, 0.0, ab.F_SCORE | ab.F_NO_RECOMPUTE, scores[i:i + 1], None, y)
    assert dc.ctx.poll_status() == 0
    assert scores[0].sum().item() > 0 and torch.equal(scores[0], scores[1])


@pytest.mark.parametrize("T", [51198, 51199])     # with the two mask words of 40 rows: the map just fits, just does not
def test_probe_row_mask_of_long_contexts(T):
    lay = wl.make_layout(1, 0, T - 40, 8, 32, 32, "all")
    case = wl.make_case(MID128, lay, 0.0, cfg_id=72)
    dc = DeviceCase(case)
    K, s_gpu, _, _ = run_layer_step(dc, 0.0, ab.F_SCORE)
    assert dc.ctx.poll_status() == 0
    ref = oracle_step(case, 0, ratio=0.0)["scores"]
    # Eq. 4-5 from bf16 products summed in fp32: the bound the other scoring tests use
    assert np.all(np.abs(s_gpu[0] - ref) <= 1e-3 * np.maximum(ref, ref.mean()))


def test_probe_scores_of_more_than_256_query_tiles():
    # 32964 rows in 258 tiles, the masked ones in the last: against the scoring kernels on the same cache (Eq. 4-5 from bf16
    # queries and keys summed in fp32: the bound the other scoring tests use)
    shape = wl.LayerShape(256, 2, 1, 128, 256, 1e-5, False, 5e5, "probe-many-rows")
    lay = wl.make_layout(1, 0, 64, 32900, 64, 32, "all")
    case = wl.make_case(shape, lay, 0.0, cfg_id=81)
    dc = DeviceCase(case)
    scores = torch.zeros((2, 64), dtype=torch.float32, device=DEV)
    y = torch.zeros((1, lay.n_extra, 256), dtype=torch.bfloat16, device=DEV)
    for i, flags in enumerate((ab.F_SCORE | ab.F_NO_RECOMPUTE, ab.F_SCORE)):
        dc.ctx.layer_step(dc.lw, dc.req, dc.kv(), dc.x, 0, 0.0, flags, scores[i:i + 1], None, y)
    assert dc.ctx.poll_status() == 0
    apart, probe = scores.cpu().numpy().astype(np.float64)
    assert apart.min() > 0 and np.all(np.abs(probe - apart) <= 1e-3 * np.maximum(apart, apart.mean()))


@pytest.mark.parametrize("L", [255, 256, 257, 1025, 2047, 8192, 16385])
def test_topk_score_distributions(L):
    """Histogram ranges and candidate counts the selection's passes depend on: a few huge scores over many small ones,
    a narrow band, zeros and denormals, more equal scores around the threshold than are ranked directly."""
    g = np.random.default_rng(L)
    ctx = ab.Context.for_shape(wl.TINY, 1, 256, 128, 1, 1, DEV)
    spread = np.exp(4.0 * g.standard_normal(L))
    narrow = 1.0 + 1e-6 * g.random(L)
    sparse = np.where(g.random(L) < 0.05, g.random(L), 0.0)
    sparse[::7] = 1e-41
    bands = np.where(g.random(L) < 0.5, 0.5, g.random(L))
    signs = g.standard_normal(L) * 1e30
    for name, s in (("spread", spread), ("narrow", narrow), ("sparse", sparse), ("bands", bands), ("signs", signs)):
        s = s.astype(np.float32)
        for K in sorted({1, L // 10, L // 2, L - 1}):
            out = torch.full((1, K), -7, dtype=torch.int32, device=DEV)
            ctx.select_topk(torch.from_numpy(s).to(DEV), 1, L, K, out)
            assert np.array_equal(out[0].cpu().numpy(), orc.select_topk(s, K)[0]), (name, L, K)


# K is cut between 1, 2 or 4 CTAs of a cluster depending on rows and shape; a ring stage takes 1 to 8 panels of K; up to 112 rows the
# cluster's parts arrive beside the ring, above in it (tiles of 128 columns over four CTAs)
DEEP128 = wl.LayerShape(3584, 4, 1, 128, 8192, 1e-6, True, 1e6, "deep-d128")
ODD64 = wl.LayerShape(1024, 6, 2, 64, 640, 1e-5, False, 5e5, "odd-d64")
DEEP64 = wl.LayerShape(2048, 12, 4, 64, 256, 1e-5, False, 5e5, "deep-d64")
# gate/up of more 256-column tiles than SMs: the general one-SM kernel, whole and cut tiles
WIDE_FFN = wl.LayerShape(256, 2, 1, 128, 19200, 1e-5, False, 5e5, "wide-ffn")
# rows of up to 256 columns: every CTA prepares them itself up to 64 rows
NARROW128 = wl.LayerShape(128, 2, 2, 64, 384, 1e-6, True, 1e6, "narrow-128")


@pytest.mark.parametrize("shape,rows", [(DEEP128, n) for n in (1, 8, 33, 103, 112, 113, 128, 129)] + [(ODD64, n) for n in (1, 7, 9, 64, 127)]
                         + [(DEEP64, n) for n in (7, 127)] + [(WIDE_FFN, n) for n in (1, 40, 64, 65, 128)]
                         + [(NARROW128, n) for n in (1, 9, 63, 64, 65)])
def test_few_row_projections(shape, rows):
    lay = wl.make_layout(1, 3, 160, 8, 8, 8, "none")
    case = wl.make_case(shape, lay, 0.0, cfg_id=73, weights=cached_weights(shape, 73))
    dc = DeviceCase(case)
    anchors = np.sort(np.random.default_rng(rows).choice(160, rows, replace=False)).astype(np.int32)[None]
    k_new, v_new, y = run_split_calls(dc, torch.from_numpy(anchors).to(DEV), rows)
    assert dc.ctx.poll_status() == 0
    check_against_oracle(dc, anchors, k_new, v_new, y, None, None, rows)


# 3, 5, 9, 17 and 40 key tiles: 1, 2, 4, 8 and 8 CTAs per query tile, with unequal shares
@pytest.mark.parametrize("T,rows,drop", [(300, 33, False), (520, 1, False), (1100, 128, True), (2100, 40, False), (5000, 97, True)])
def test_attention_key_split(T, rows, drop):
    lay = wl.make_layout(1, 6, T - 6 - 40, 8, 32, 32, "none")
    case = wl.make_case(MID128, lay, 0.0, cfg_id=74)
    dc = DeviceCase(case, max_rows=rows)
    ratio = (rows - 0.5) / lay.affix_len
    anchors = np.sort(np.random.default_rng(T).choice(lay.affix_len, rows, replace=False)).astype(np.int32)[None]
    _, _, _, y = run_layer_step(dc, ratio, ab.F_DROP_NON_ANCHOR if drop else 0, anchors)
    assert dc.ctx.poll_status() == 0
    ref = oracle_step(case, 0, anchor_idx=anchors[0], drop_non_anchor=drop)
    assert_close_bf16(ab.to_host_bits(y[0]), ref["y"], "y")


# rows that no longer fit a warp's registers in the row preparation
WIDE128 = wl.LayerShape(5376, 2, 1, 128, 256, 1e-5, False, 5e5, "wide-d128")
# K long enough for few tiles to be cut between clusters, in the q/k/v and the gate/up projection
LONGK128 = wl.LayerShape(3584, 4, 1, 128, 1024, 1e-6, True, 1e6, "longk-d128")
# an odd number of 128-column units: the last weight tile is half past the end of the row, whole or cut
ODD_TILES = wl.LayerShape(1920, 2, 1, 128, 256, 1e-5, False, 5e5, "odd-tiles")


@pytest.mark.parametrize("shape,rows", [(ODD_TILES, n) for n in (9, 128, 140, 300)]
                         + [(MID128, 129), (MID128, 257), (MID128, 600), (WIDE128, 140), (WIDE128, 300)]
                         + [(LONGK128, 129), (LONGK128, 385)])
def test_row_counts_of_wide_shapes(shape, rows):
    lay = wl.make_layout(1, 3, rows + 40, 8, 8, 8, "none")
    case = wl.make_case(shape, lay, 0.0, cfg_id=75)
    dc = DeviceCase(case, max_rows=rows)
    anchors = np.sort(np.random.default_rng(rows).choice(lay.affix_len, rows, replace=False)).astype(np.int32)[None]
    k_new, v_new, y = run_split_calls(dc, torch.from_numpy(anchors).to(DEV), rows)
    assert dc.ctx.poll_status() == 0
    check_against_oracle(dc, anchors, k_new, v_new, y, None, None, rows)


# a few keys four times as long, so that the exponents' reference moves on a later key tile: one CTA and a cluster per query
# tile, with and without masked keys
@pytest.mark.parametrize("T,rows,drop", [(1100, 40, False), (1100, 40, True), (700, 200, True), (4500, 300, False)])
def test_attention_reference_moves(T, rows, drop):
    lay = wl.make_layout(1, 6, T - 6 - 40, 8, 32, 32, "none")
    case = wl.make_case(MID128, lay, 0.0, cfg_id=76, hot_frac=0.01)
    dc = DeviceCase(case, max_rows=rows)
    ratio = (rows - 0.5) / lay.affix_len
    anchors = np.sort(np.random.default_rng(T).choice(lay.affix_len, rows, replace=False)).astype(np.int32)[None]
    _, _, _, y = run_layer_step(dc, ratio, ab.F_DROP_NON_ANCHOR if drop else 0, anchors)
    assert dc.ctx.poll_status() == 0
    ref = oracle_step(case, 0, anchor_idx=anchors[0], drop_non_anchor=drop)
    assert_close_bf16(ab.to_host_bits(y[0]), ref["y"], "y")


# many more (query tile, head, request) items than SMs: several per CTA, the last round incomplete; query tiles with empty
# quarters; and over a shared cache four requests to a tile, an item per CTA, with a last group of two
HEADS32 = wl.LayerShape(256, 32, 4, 128, 256, 1e-5, False, 5e5, "heads32")


@pytest.mark.parametrize("B,T,rows,shared", [(30, 300, 40, False), (15, 4200, 203, False), (118, 160, 9, True)])
def test_attention_items_per_cta(B, T, rows, shared):
    lay = wl.make_layout(B, 3, T - 27, 8, 8, 8, "none")
    case = wl.make_case(HEADS32, lay, 0.0, cfg_id=77, weights=cached_weights(HEADS32, 77))
    dc = DeviceCase(case, max_rows=rows)
    rng = np.random.default_rng(T)
    anchors = np.stack([np.sort(rng.choice(lay.affix_len, rows, replace=False)) for _ in range(B)]).astype(np.int32)
    da = torch.from_numpy(anchors).to(DEV)
    if shared:
        dsk, dsv = ab.to_device_bf16(case.cache_k[:1].copy(), DEV), ab.to_device_bf16(case.cache_v[:1].copy(), DEV)
        k_new = torch.zeros((B, rows, 4, 128), dtype=torch.bfloat16, device=DEV)
        v_new, y = torch.zeros_like(k_new), torch.zeros((B, rows, 256), dtype=torch.bfloat16, device=DEV)
        dc.ctx.recompute_anchors(dc.lw, dc.req, ab.KV(dsk.data_ptr(), dsv.data_ptr(), 0, T), dc.x, 0, da, rows, k_new, v_new, y)
    else:
        y = run_layer_step(dc, (rows - 0.5) / lay.affix_len, 0, anchors)[3]
    assert dc.ctx.poll_status() == 0
    for b in (0, 1, B // 2, B - 1):
        c = 0 if shared else b
        ref = orc.layer_step(case.weights, HEADS32, case.x[b], case.cache_k[c], case.cache_v[c], T, lay.affix_start, lay.affix_len,
                             lay.masked_pos[b], lay.extra_rows[b], case.rope_cos, case.rope_sin, anchor_idx=anchors[b])
        assert_close_bf16(ab.to_host_bits(y[b]), ref["y"], "y")


# Decode passes over a shared cache, private rows in rounds behind the shared tiles: groups of four in clusters of 4, 2, 8 and 8 CTAs
# (some without a step of their own), a pair on one CTA (the third case), and one request to a tile in clusters of 8 and 4 (the fourth
# and the last).  Groups that are not full; an affix that neither starts nor ends with a tile.
@pytest.mark.parametrize("shape,B,pre,L,post,rows,ratio", [
    (HEADS32, 4, 0, 300, 40, 32, 0.3), (HEADS32, 6, 150, 500, 180, 7, 0.5), (HEADS32, 5, 5, 260, 90, 64, 0.2),
    (MID128, 2, 9, 700, 60, 33, 0.2), (MID128, 3, 300, 200, 300, 20, 0.1), (MID128, 2, 0, 2500, 64, 1, 0.05),
    (MID128, 7, 130, 1100, 100, 50, 0.35)])
def test_attention_of_grouped_requests(shape, B, pre, L, post, rows, ratio):
    lay = wl.make_layout(B, pre, L, post, rows, rows, "all")
    case = wl.make_case(shape, lay, ratio, cfg_id=78, weights=cached_weights(shape, 78), hot_frac=0.01)
    T, K = lay.ctx_len, orc.k_from_ratio(L, ratio)
    dc = DeviceCase(case, max_rows=K + lay.n_extra)
    rng = np.random.default_rng(T)
    anchors = np.stack([np.sort(rng.choice(L, K, replace=False)) for _ in range(B)]).astype(np.int32)
    own = np.concatenate([anchors + pre, lay.extra_rows], axis=1)              # position of every private row
    where = [{int(p): i for i, p in enumerate(own[b])} for b in range(B)]
    slot_rows = np.stack([[where[b][int(p)] for p in lay.masked_pos[b]] for b in range(B)]).astype(np.int32)
    on = lambda t: torch.from_numpy(np.ascontiguousarray(t)).to(DEV)
    shared = [ab.to_device_bf16(c[:1].copy(), DEV) for c in (case.cache_k, case.cache_v)]
    mine = [c[np.arange(B)[:, None], own] for c in (case.cache_k, case.cache_v)]
    k_slots, v_slots = (ab.to_device_bf16(np.ascontiguousarray(m), DEV) for m in mine)
    block = on(lay.masked_pos)
    req = ab.Context.request(B, T, pre, L, block, block, dc.cos, dc.sin)
    y = torch.zeros((B, rows, shape.hidden), dtype=torch.bfloat16, device=DEV)
    dc.ctx.recompute_rows_shared(dc.lw, req, dc.req, ab.KV(shared[0].data_ptr(), shared[1].data_ptr(), 0, T), dc.x, 0, on(anchors), K,
                                 on(slot_rows), k_slots, v_slots, y)
    assert dc.ctx.poll_status() == 0
    for b in {0, 1, B // 2, B - 1}:
        ck, cv = case.cache_k[0].copy(), case.cache_v[0].copy()
        ck[own[b]], cv[own[b]] = mine[0][b], mine[1][b]
        ref = orc.layer_step(case.weights, shape, case.x[b], ck, cv, T, pre, L, lay.masked_pos[b], lay.masked_pos[b], case.rope_cos,
                             case.rope_sin, anchor_idx=np.zeros(0, np.int32))
        assert_close_bf16(ab.to_host_bits(y[b]), ref["y"], "y")


# One CTA per query tile, which leaves out the shared tiles without a key: two in front of the affix, one or more behind it, several
# private rounds.  Groups of four, two and three of them part-filled; pairs; one request to a tile; two tiles of one request.
UNSPLIT = {"attention_group_kernel": [(HEADS32, 12, 300, 300, 150, 20, 0.2), (HEADS32, 9, 290, 200, 140, 31, 0.5),
                                      (HEADS32, 6, 300, 260, 290, 50, 0.2), (HEADS32, 5, 270, 270, 150, 33, 0.2)],
           "attention_tc_kernel<false>": [(HEADS32, 3, 300, 260, 150, 70, 0.2)],
           "attention_tc2q_kernel": [(HEADS32, 5, 300, 260, 150, 140, 0.2)]}


@pytest.mark.parametrize("kernel", UNSPLIT)
def test_attention_without_the_empty_tiles_of_a_shared_cache(kernel):
    asked = [(shape, B, pre, L, post, rows, orc.k_from_ratio(L, ratio)) for shape, B, pre, L, post, rows, ratio in UNSPLIT[kernel]]
    for case, kernels in zip(UNSPLIT[kernel], launched_kernels(asked, "shared_decode")):
        assert kernel in kernels and kernels.count("attention") == kernels.count(kernel), (case, kernels)
        test_attention_of_grouped_requests(*case)


# Two requests of 33 to 64 rows share a tile where that saves rounds of CTAs (on 148 SMs): 2 | 1, 3 | 2, 5 | 3 rounds, but not 1 | 1
# nor 2 | 2.  Up to 32 rows four always do; more than 64 never.
def test_which_decode_passes_share_query_tiles():
    cases = [(5, 48, 1), (9, 48, 0), (9, 33, 0), (9, 64, 0), (10, 48, 1), (13, 64, 1), (19, 33, 1), (4, 48, 0), (4, 32, 1), (9, 32, 1),
             (2, 7, 1), (10, 65, 0)]
    launched = launched_kernels([(HEADS32, B, 5, 150, 20, rows, 10) for B, rows, _ in cases], "shared_decode")
    for (B, rows, grouped), kernels in zip(cases, launched):
        assert ("attention_group_kernel" in kernels) == bool(grouped), (B, rows, kernels)
        assert ("attention_tc_kernel<false>" in kernels) != bool(grouped), (B, rows, kernels)


# One-pass scoring with three CTAs per SM: one CTA per (request, head) and clusters of two, four and eight; 2 to 4 key tiles per CTA, the
# last one ragged; 1 to 32 masked rows; both normalisers; one cache for the batch.
THREE_CTAS = [(HEADS32, 10, 300, 32, False, False), (HEADS32, 12, 385, 29, False, True), (HEADS32, 5, 700, 29, True, False),
              (HEADS32, 3, 1500, 1, False, False), (MID128, 10, 3990, 30, False, True), (MID128, 10, 3990, 17, True, False)]


def test_scoring_with_three_ctas_per_sm():
    launched = launched_kernels([(s, B, L, m, shared, norm_full) for s, B, L, m, shared, norm_full in THREE_CTAS], "scoring")
    for case, kernels in zip(THREE_CTAS, launched):
        assert "score_onepass_tc_kernel<32, 2, 3>" in kernels, (case, kernels)
    for shape, B, L, m, shared, norm_full in THREE_CTAS:
        lay = wl.make_layout(B, 7, L, 20, max(m, 8), m)
        ck, q = wl.random_kv_cache(shape, lay, 83)[0], wl.random_q_mask(shape, lay, 84)
        dk, dq = ab.to_device_bf16(ck, DEV), ab.to_device_bf16(q, DEV)
        masked = torch.from_numpy(lay.masked_pos.copy()).to(DEV)
        ctx = ab.Context.for_shape(shape, B, lay.ctx_len, L, 1, m, DEV)
        req = ab.Context.request(B, lay.ctx_len, 7, L, masked, None, None, None)
        scores = torch.zeros((B, L), dtype=torch.float32, device=DEV)
        kv = ab.KV(dk.data_ptr(), dk.data_ptr(), 0, lay.ctx_len) if shared else ab.Context.kv(dk, dk)
        ctx.score_anchors(req, dq, kv, scores, accumulate=False, norm_full=norm_full)
        assert ctx.poll_status() == 0
        for b in (0, B // 2, B - 1):
            keys = orc.bf16_bits_to_f64(ck[0 if shared else b, :lay.ctx_len])
            ref = orc.score_anchors(orc.bf16_bits_to_f64(q[b]), keys[7:7 + L], keys, 7, norm_full)
            got = scores[b].cpu().numpy().astype(np.float64)
            assert (np.abs(got - ref) / np.maximum(ref, ref.mean())).max() < 1e-3, (shape.name, B, L, m)


# Small projections sum K in the general kernel's order, block by block: a row's bits do not depend on how many rows are in the
# call, on the tile or on the split over a cluster (140 rows take the two-SM kernel).  Every product is reached with inputs that
# the other rows of a call do not change: no queries, hence equal weights over equal values, so that the attention's output is
# the bias of V exactly.
NARROW512 = wl.LayerShape(512, 2, 1, 128, 512, 1e-6, True, 1e6, "narrow-512")       # eight blocks: q/k/v over two CTAs
NARROW1K = wl.LayerShape(1024, 1, 1, 128, 384, 1e-6, True, 1e6, "narrow-1k")        # sixteen: q/k/v on the general kernel


@pytest.mark.parametrize("shape,counts", [(wl.TINY_GQA, (1, 9, 60, 128)), (NARROW512, (40, 57, 128)), (NARROW1K, (49, 128))])
def test_small_projections_do_not_depend_on_the_number_of_rows(shape, counts):
    lay = wl.make_layout(1, 3, 200, 8, 8, 8, "none")
    case = wl.make_case(shape, lay, 0.0, cfg_id=78)
    w = dict(case.weights)
    for name in ("wq", "bq", "wv"):
        w[name] = np.zeros_like(w[name])
    w["bv"] = orc.f64_to_bf16_bits(np.random.default_rng(78).standard_normal(w["bv"].shape))
    case.weights = w
    case.cache_v[:] = w["bv"].reshape(case.cache_v.shape[2:])
    dc = DeviceCase(case, max_rows=140)
    rows = np.sort(np.random.default_rng(79).choice(200, 140, replace=False)).astype(np.int32)

    def outputs(anchors):
        k_new, v_new, y = run_split_calls(dc, torch.from_numpy(anchors[None].copy()).to(DEV), len(anchors))
        assert dc.ctx.poll_status() == 0
        assert torch.equal(v_new[0], dc.cv[0, :len(anchors)])
        return k_new[0], y[0]

    k_all, y_all = outputs(rows)
    for n in counts:
        pick = np.sort(np.random.default_rng(n).choice(140, n, replace=False))
        k_new, y = outputs(rows[pick])
        at = torch.from_numpy(pick).to(DEV)
        assert torch.equal(k_new, k_all[at]) and torch.equal(y, y_all[at]), n


# With 256 columns of K, gate/up of these row counts fills 43, 54 and 65 % of a wave with pair tiles: cut, hence with a finish
# kernel, in all three (whole tiles would add the K blocks in another order).
def test_short_contractions_are_cut_up_to_two_thirds_of_a_wave():
    lay = wl.make_layout(1, 3, 1500, 8, 8, 8, "none")
    case = wl.make_case(wl.TINY, lay, 0.0, cfg_id=80)
    launches = []
    for rows in (1000, 1100, 1500):
        dc = DeviceCase(case, max_rows=rows)
        anchors = np.sort(np.random.default_rng(rows).choice(1500, rows, replace=False)).astype(np.int32)[None]
        k_new, v_new, y = run_split_calls(dc, torch.from_numpy(anchors).to(DEV), rows)
        assert dc.ctx.poll_status() == 0
        check_against_oracle(dc, anchors, k_new, v_new, y, None, None, rows)
        launches.append(dc.ctx.launch_count())
    assert launches[0] == launches[1] == launches[2]


# Whole tiles with the weights as the product's M (gemm_wm_kernel), both rotary orders, biases and grouped heads, w_up in memory above
# and below w_gate, the residual epilogue in the WIDE shapes.  256 columns: fewer K blocks than ring stages, chunks of 64 to 144
# rows, the last one part-filled or full (288); where chunks save too little, whole tiles.  1024 columns: the ring wraps; 140 rows are
# one chunk of 144, 540 rows four, three tiles to a cluster, so that an accumulator is taken again.
WM128 = wl.LayerShape(256, 40, 5, 128, 3328, 1e-5, True, 5e5, "wm-d128")
WM64 = wl.LayerShape(256, 80, 10, 64, 3328, 1e-5, True, 5e5, "wm-d64")
WM_WIDE = wl.LayerShape(6400, 2, 1, 128, 256, 1e-5, False, 5e5, "wm-wide")
WM128_DEEP = wl.LayerShape(1024, 92, 4, 128, 6400, 1e-5, True, 5e5, "wm-d128-deep")
WM64_DEEP = wl.LayerShape(1024, 184, 8, 64, 6400, 1e-5, True, 5e5, "wm-d64-deep")
WM_WIDE_DEEP = wl.LayerShape(12800, 8, 1, 128, 1024, 1e-5, True, 5e5, "wm-wide-deep")
WM_CASES = [(WM128, 280, False), (WM128, 288, True), (WM128, 333, True), (WM128, 545, False), (WM64, 260, True), (WM64, 300, False),
            (WM64, 417, False), (WM_WIDE, 257, False), (WM_WIDE, 400, False), (WM_WIDE, 545, False), (WM128_DEEP, 140, True),
            (WM128_DEEP, 540, False), (WM64_DEEP, 140, False), (WM64_DEEP, 540, True)]
WM_TOO_LITTLE = [(WM128, 333), (WM64, 417), (WM_WIDE, 400)]


def wm_case(shape, rows, max_rows, up_first):
    lay = wl.make_layout(1, 3, max_rows + 30, 8, 8, 8, "none")
    case = wl.make_case(shape, lay, 0.0, cfg_id=81, weights=cached_weights(shape, 81))
    dc = DeviceCase(case, max_rows=max_rows)
    order = ("w_up", "w_gate") if up_first else ("w_gate", "w_up")
    both = torch.stack([dc.w_dev[n] for n in order])
    for i, n in enumerate(order):
        dc.w_dev[n] = both[i]
    dc.lw = ab.Context.weights(dc.w_dev)
    return dc, np.sort(np.random.default_rng(rows).choice(lay.affix_len, max_rows, replace=False)).astype(np.int32)


def wm_split_calls(dc, anchors):
    out = run_split_calls(dc, torch.from_numpy(anchors[None].copy()).to(DEV), len(anchors))
    assert dc.ctx.poll_status() == 0
    return out


# The next two tests compare results; this one says that the kernel they mean is the one that runs.  Gate/up with few K blocks is
# bound by its epilogue, which is the longer one with the weights as M, whatever the chunks save: the last two.
def test_which_projections_take_the_weights_as_m():
    short = [(wl.TINY, 2045), (wl.LayerShape(1024, 2, 1, 128, 3072, 1e-5, False, 5e5, "gate-up-1k"), 615)]
    whole = [(s, n) for s in (WM128_DEEP, WM64_DEEP, WM_WIDE_DEEP) for n in (256, 768)] + WM_TOO_LITTLE + short
    taken = [c[:2] for c in WM_CASES if c[:2] not in WM_TOO_LITTLE] + [(s, n) for s in (WM128_DEEP, WM64_DEEP, WM_WIDE_DEEP) for n in (150, 540)]
    launched = launched_kernels(taken + whole)
    for (shape, rows), kernels in zip(taken, launched):
        for epilogue in (1,) if shape in (WM_WIDE, WM_WIDE_DEEP) else (0, 2):            # residual; q/k/v and gate/up
            assert f"gemm_wm_kernel<{epilogue}>" in kernels, (shape.name, rows, kernels)
    for (shape, rows), kernels in zip(whole, launched[len(taken):]):
        assert "gemm_tc2_kernel" in kernels and "gemm_wm_kernel" not in kernels, (shape.name, rows, kernels)


@pytest.mark.parametrize("shape,rows,up_first", WM_CASES)
def test_weights_as_m_projections(shape, rows, up_first):
    dc, anchors = wm_case(shape, rows, rows, up_first)
    check_against_oracle(dc, anchors[None], *wm_split_calls(dc, anchors), None, None, rows)


# The same rows at the head of a call of whole 256 x 256 tiles have the same bits (as many row pairs, so that cut projections are cut
# alike).  k_new and v_new as they are; y with inputs that the other rows do not change (as above: no queries, equal values).
@pytest.mark.parametrize("shape,up_first", [(WM128_DEEP, False), (WM64_DEEP, True), (WM_WIDE_DEEP, False)])
@pytest.mark.parametrize("rows,more", [(150, 256), (540, 768)])
def test_weights_as_m_projections_have_the_bits_of_whole_tiles(shape, up_first, rows, more):
    dc, anchors = wm_case(shape, rows, more, up_first)
    few, many = wm_split_calls(dc, anchors[:rows]), wm_split_calls(dc, anchors)
    assert torch.equal(few[0], many[0][:, :rows]) and torch.equal(few[1], many[1][:, :rows])
    for name in ("wq", "bq", "wv"):
        dc.w_dev[name].zero_()
    dc.cv[:] = dc.w_dev["bv"].view(shape.n_kv_heads, shape.head_dim)
    few, many = wm_split_calls(dc, anchors[:rows]), wm_split_calls(dc, anchors)
    assert torch.equal(few[1][0], dc.cv[0, :rows])
    assert torch.equal(few[2], many[2][:, :rows])
