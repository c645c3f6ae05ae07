"""Sizes at which the kernels of middle decode batches and of the largest prefill passes can go wrong: 32-token units and
pages that begin or end with the newest token, (row, head) pairs cut over warps, row tiles without rows, ragged tiles;
each against the fp64 oracle on identical history."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from oracle import gpt_oracle as O
from paper_2607_21042_b200 import binding as B
from paper_2607_21042_b200 import cases as C
from helpers import E4M3_MAX_ABS, E4M3_REL_L2, E4M3_REL_L2_SHORT, assert_logits_close, bits_dev, check_tokens, logits_errors

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _run(eng, prefixes, n_steps, **kw):
    S, V = len(prefixes), eng.cfg.vocab
    toks = torch.zeros((n_steps + 1, S), dtype=torch.int32, device=DEV)
    logits = torch.zeros((n_steps + 1, S, V), dtype=torch.float32, device=DEV)
    ids, _ = eng.prefill([bits_dev(p) for p in prefixes], out_tokens=toks[0], out_logits=logits[0], **kw)
    for k in range(1, n_steps + 1):
        eng.decode_step(ids, toks[k], out_logits=logits[k], **kw)
    eng.sync()
    for s in ids:
        eng.release_stream(s)
    return logits.cpu().numpy().transpose(1, 0, 2), toks.cpu().numpy().T


def _check(model, prefixes, lg, tk, streams, what):
    for s in streams:
        ref, _ = O.replay_full(model, O.bf16_to_f64(prefixes[s]), tk[s][:-1])
        assert_logits_close(lg[s], ref, "%s, stream %d" % (what, s))
        check_tokens(tk[s], ref, 0, 1.0, None, "%s, stream %d" % (what, s))


def _check_e4m3(model, prefixes, lg, tk, streams, what):
    """The bars of the 8-bit cache: the relative one is wider below 32 attended tokens (see helpers)."""
    for s in streams:
        ref, _ = O.replay_full(model, O.bf16_to_f64(prefixes[s]), tk[s][:-1])
        ctx = prefixes[s].shape[0] + np.arange(len(ref))
        for i in range(len(ref)):
            ma, rl = logits_errors(lg[s][i], ref[i])
            bar = E4M3_REL_L2 if ctx[i] >= 32 else E4M3_REL_L2_SHORT
            assert ma <= E4M3_MAX_ABS and rl <= bar, "%s, stream %d, step %d: max-abs %.4g, relative L2 %.4g" % (what, s, i, ma, rl)


@pytest.mark.parametrize("S", [75, 100, 128])
def test_unit_split_decode_attention(S):
    """300, 400 and 512 (row, head) pairs on one CTA per SM: contexts that cross 32-token and page edges while they decode,
    one long context among short ones, stale pages full of NaN behind every context."""
    edges = [1, 30, 31, 32, 33, 62, 63, 64, 65, 95, 96, 127, 128, 700]
    lens = [edges[i % len(edges)] if i < 28 else 2 + (11 * i) % 60 for i in range(S)]
    cfg = C.tiny_config(max_streams=S, n_pages=sum((x + 8 + 63) // 64 for x in lens), max_context=768)
    w = C.make_weights(cfg, seed=21)
    model = O.OracleModel(cfg, w)
    eng = B.TtsGpt(cfg, w, DEV)
    eng.set_option("poison_free_pages", 1)
    prefixes = C.make_prefixes(cfg, lens, seed=22)
    lg, tk = _run(eng, prefixes, 4)
    _check(model, prefixes, lg, tk, list(range(14)) + [S - 1], "unit-split attention")
    lg2, _ = _run(eng, prefixes, 4)
    assert np.array_equal(lg, lg2)
    eng.set_option("attn_decode", 0)      # one CTA per pair
    lg3, _ = _run(eng, prefixes, 4)
    assert np.max(np.abs(lg3[:, :2] - lg[:, :2])) < 3e-2
    eng.destroy()


@pytest.mark.parametrize("wfmt", [C.W_BF16, C.W_INT8_PC, C.W_INT4_G128])
@pytest.mark.parametrize("S,d", [(2, 1280), (5, 384), (7, 256), (10, 1280), (6, 1152)])
def test_layernorm_fused_into_linears_of_several_rows(S, d, wfmt):
    """A warp per row in every CTA (2, 3 and 10 float4 per lane), FC2's k-ranges added up by a cluster (shares that do and do not
    divide evenly), hidden rows from the fused head; against the oracle, and against LayerNorm kernels of their own."""
    cfg = C.tiny_config(d_model=d, n_head=d // 64, d_ff=4 * d if d < 1280 else 1536, wfmt=wfmt, max_streams=S, n_pages=3 * S)
    w = C.make_weights(cfg, seed=53)
    model = O.OracleModel(cfg, w)
    eng = B.TtsGpt(cfg, w, DEV)
    prefixes = C.make_prefixes(cfg, [20 + 9 * i for i in range(S)], seed=54)
    hid = torch.zeros((2, S, d), dtype=torch.bfloat16, device=DEV)
    lg, tk = _run(eng, prefixes, 3, out_hidden=hid[0])
    _check(model, prefixes, lg, tk, range(S), "fused LayerNorm")
    assert np.array_equal(lg, _run(eng, prefixes, 3)[0])
    eng.set_option("ln_fuse_rows", 1)
    lg2, tk2 = _run(eng, prefixes, 3, out_hidden=hid[1])
    _check(model, prefixes, lg2, tk2, range(S), "LayerNorm kernels")
    # rows of unit variance whose bf16 operands round along two orders of sums: a few bf16 steps (2^-8 of a value), one in the mean
    same = np.array([np.array_equal(a, b) for a, b in zip(tk, tk2)])
    a, b = hid[0].float().cpu().numpy()[same], hid[1].float().cpu().numpy()[same]
    assert same.any() and np.linalg.norm(a - b) <= 2.0 ** -7 * np.linalg.norm(a)
    assert eng.check_canaries() == 0
    eng.destroy()


@pytest.mark.parametrize("S,d,wfmt,kv,fused", [
    (7, 1280, C.W_BF16, C.KV_BF16, True), (8, 1280, C.W_BF16, C.KV_BF16, False), (10, 1280, C.W_INT8_PC, C.KV_BF16, False), (8, 1280, C.W_INT4_G128, C.KV_BF16, True),
    (8, 1280, C.W_BF16, C.KV_FP8_E4M3, True), (8, 1024, C.W_INT8_PC, C.KV_BF16, True), (10, 256, C.W_BF16, C.KV_BF16, True), (11, 256, C.W_BF16, C.KV_BF16, False)])
def test_rule_of_the_fused_layernorm(S, d, wfmt, kv, fused):
    """Steps on either side of the rule's lines have the bits of the form it names, and those of the other form (up to 16 rows: two
    per warp) pass the oracle's bars too."""
    cfg = C.tiny_config(d_model=d, n_head=d // 64, d_ff=1536, wfmt=wfmt, kv_fmt=kv, max_streams=S, n_pages=3 * S)
    w = C.make_weights(cfg, seed=63)
    model = O.OracleModel(cfg, w)
    prefixes = C.make_prefixes(cfg, [40 + 5 * i for i in range(S)], seed=64)
    out = {}
    for rows in (None, 1, 16):
        eng = B.TtsGpt(cfg, w, DEV)
        if rows:
            eng.set_option("ln_fuse_rows", rows)
        out[rows] = _run(eng, prefixes, 3)
        (_check_e4m3 if kv == C.KV_FP8_E4M3 else _check)(model, prefixes, *out[rows], range(S), "ln_fuse_rows %s" % rows)
        eng.destroy()
    assert np.array_equal(out[None][0], out[16 if fused else 1][0])
    assert not np.array_equal(out[1][0], out[16][0])


@pytest.mark.parametrize("wfmt,S,d,cols", [(C.W_BF16, 5, 256, 8), (C.W_INT8_PC, 10, 1280, 24), (C.W_INT4_G128, 2, 1280, 24)])
def test_a_cluster_stores_nothing_behind_an_expired_wait(wfmt, S, d, cols):
    """The weights of one k-range do not arrive: its cluster's columns (one and three 8-row tiles per CTA) are not stored by any of its
    CTAs, all others are whole, the error is reported once and the engine goes on."""
    cfg = C.tiny_config(d_model=d, n_head=d // 64, d_ff=4 * d, wfmt=wfmt, max_streams=S, n_pages=2 * S)
    eng = B.TtsGpt(cfg, C.make_weights(cfg, seed=67), DEV)
    prefixes = C.make_prefixes(cfg, [7 + i for i in range(S)], seed=68)
    lg, tk = _run(eng, prefixes, 2)
    _run(eng, prefixes, 1, top_k=4, uniforms=torch.zeros(S, device=DEV))   # a sampled call in front changes nothing here
    mark = torch.arange(S * d, device=DEV, dtype=torch.float32).view(S, d) / 7
    whole, out = mark.clone(), mark.clone()
    eng.wait_for_caller()
    eng.debug_expire_linear(3, S, -1, 1000, whole)
    eng.sync()
    assert not bool((whole == mark).all(0).any()) and bool(torch.isfinite(whole).all())
    eng.debug_expire_linear(3, S, 2, 1000, out)
    with pytest.raises(B.TtsGptError) as e:
        eng.sync()
    assert e.value.code == B.E_TIMEOUT
    lost = torch.zeros(d, dtype=torch.bool, device=DEV)
    lost[2 * cols:3 * cols] = True
    assert torch.equal(out[:, lost], mark[:, lost]) and torch.equal(out[:, ~lost], whole[:, ~lost])
    eng.sync()
    lg2, tk2 = _run(eng, prefixes, 2)
    assert np.array_equal(lg, lg2) and np.array_equal(tk, tk2)
    eng.destroy()


@pytest.mark.parametrize("wfmt,S,d_ff", [(C.W_BF16, 10, 8832), (C.W_BF16, 10, 8960), (C.W_BF16, 9, 10240), (C.W_INT8_PC, 10, 10240), (C.W_INT4_G128, 10, 10240)])
def test_fc2_whose_rows_do_not_fit_a_cluster(wfmt, S, d_ff):
    """Small batches on either side of the longest K whose staged rows a cluster holds, in decode steps and in a prefill pass
    of as many rows."""
    cfg = C.tiny_config(d_ff=d_ff, wfmt=wfmt, max_streams=S, n_pages=2 * S)
    w = C.make_weights(cfg, seed=55)
    model = O.OracleModel(cfg, w)
    eng = B.TtsGpt(cfg, w, DEV)
    for lens in ([1] * S, [5 + i for i in range(S)]):   # the first: a pass of S rows
        prefixes = C.make_prefixes(cfg, lens, seed=56)
        lg, tk = _run(eng, prefixes, 3)
        _check(model, prefixes, lg, tk, range(S), "FC2 of K = %d" % d_ff)
    assert eng.check_canaries() == 0
    eng.destroy()


@pytest.mark.parametrize("S", [2, 45, 80, 128])
def test_queued_attention_has_the_bits_of_a_cta_per_pair(S):
    """40 pairs on 20 CTAs (all handed out by position), 900, 1600 and 2560 on 444 (12, 712 and 1672 taken from the counter): pages
    with one token and with 64, rows whose warps have no page, a long context among short ones, several launches on one
    counter; greedy and sampled, whose steps of more than ten pairs per SM come to the queue by the rule."""
    edges = [700, 1, 63, 64, 65, 127, 128, 129, 255, 256, 257, 320]
    lens = [edges[i] if i < 12 else 2 + (37 * i) % 300 for i in range(S)]
    cfg = C.tiny_config(d_model=1280, n_head=20, d_ff=1536, max_streams=S, n_pages=sum((x + 8 + 63) // 64 for x in lens), max_context=768)
    w = C.make_weights(cfg, seed=51)
    model = O.OracleModel(cfg, w)
    eng = B.TtsGpt(cfg, w, DEV)
    prefixes = C.make_prefixes(cfg, lens, seed=52)
    u = torch.full((S,), 0.4, device=DEV)
    trace = torch.zeros(8 * eng.set_trace(None), dtype=torch.int64, device=DEV)

    def run(queue, **kw):   # logits, tokens, and in how many kernels of a step CTA 0 left a mark that of the attention only the queue's does
        if queue is not None:
            eng.set_option("attn_queue", queue)
        lg, tk = _run(eng, prefixes, 4, **kw)
        out = torch.zeros(S, dtype=torch.int32, device=DEV)
        ids, _ = eng.prefill([bits_dev(p) for p in prefixes], out_tokens=out, **kw)
        eng.set_trace(trace)
        trace.zero_()
        eng.wait_for_caller()
        eng.decode_step(ids, out, **kw)
        eng.sync()
        eng.set_trace(None)
        for s in ids:
            eng.release_stream(s)
        return lg, tk, int((trace.view(-1, 8)[:, 4] != 0).sum())

    by_rule = run(None, top_k=30, uniforms=u)
    eng.set_option("poison_free_pages", 1)
    sampled = [run(q, top_k=30, uniforms=u) for q in (0, 1)]
    for x in (by_rule, sampled[1]):
        assert np.array_equal(x[0], sampled[0][0]) and np.array_equal(x[1], sampled[0][1])
        assert x[2] == sampled[0][2] + (cfg.n_layer if 20 * S > 10 * 148 else 0)
    for name, value in (("attn_decode", 0), ("attn_half", 0), ("attn_stream_min_pairs", 1)):
        eng.set_option(name, value)
    single, queued = run(0), run(2)
    _check(model, prefixes, queued[0], queued[1], list(range(min(S, 4))) + [S - 1], "queued attention")
    assert np.array_equal(single[0], queued[0]) and np.array_equal(single[1], queued[1])
    assert queued[2] == single[2] + cfg.n_layer
    assert np.array_equal(run(0, top_k=30, uniforms=u)[0], run(2, top_k=30, uniforms=u)[0])
    assert eng.check_canaries() == 0
    eng.destroy()


@pytest.mark.parametrize("wfmt", [C.W_BF16, C.W_INT8_PC, C.W_INT4_G128])
@pytest.mark.parametrize("lens", [[1025], [700, 3, 450, 128, 1], [1279, 1281, 5, 31]])
def test_prefill_passes_of_the_pair_kernel(wfmt, lens):
    """Passes of more than 1024 rows: an odd number of row tiles (a pair whose second tile has no rows), tiles of one row,
    streams that end inside a tile; then decode steps over the pages they wrote."""
    S = len(lens)
    cfg = C.tiny_config(wfmt=wfmt, max_streams=S, n_pages=S * 22, max_context=1408, max_pos=1408)
    w = C.make_weights(cfg, seed=23)
    model = O.OracleModel(cfg, w)
    eng = B.TtsGpt(cfg, w, DEV)
    prefixes = C.make_prefixes(cfg, lens, seed=24)
    lg, tk = _run(eng, prefixes, 3)
    _check(model, prefixes, lg, tk, range(S), "pair kernel")
    assert eng.check_canaries() == 0
    eng.destroy()


@pytest.mark.parametrize("wfmt", [C.W_BF16, C.W_INT4_G128])
@pytest.mark.parametrize("kernel,rows,tile", [(0, 17, 0), (0, 128, 5), (1, 256, 4), (2, 200, 0), (2, 200, 2), (2, 256, 3), (2, 100, 5)])
def test_tensor_core_linears_store_nothing_behind_an_expired_wait(wfmt, kernel, rows, tile):
    """The warps that issue a tile's instructions give up: that tile is not stored (by either CTA of a pair), nor are a
    pair's later ones; all others are whole, the error is reported once and the engine goes on (20 k-chunks: the rings wrap).
    int4: the kernels that scale group sums, and the pair kernel on dequantized images."""
    cfg = C.tiny_config(d_model=1280, n_head=20, d_ff=1280, wfmt=wfmt, max_streams=1, n_pages=8)   # QKV: 30 tiles, 20 k-chunks
    eng = B.TtsGpt(cfg, C.make_weights(cfg, seed=33), DEV)
    if wfmt == C.W_INT4_G128 and kernel < 2:
        eng.set_option("w4_tc_exact", 1)
    prefix = C.make_prefixes(cfg, [256], seed=34)
    lg, tk = _run(eng, prefix, 0)
    mark = -12345.0
    whole = torch.full((rows, 3840), mark, device=DEV)
    out = torch.full((rows, 3840), mark, device=DEV)
    torch.cuda.synchronize()
    eng.debug_expire_linear(kernel, rows, -1, 1000, whole)
    eng.sync()
    assert not bool((whole == mark).any()) and bool(torch.isfinite(whole).all())
    eng.debug_expire_linear(kernel, rows, tile, 1000, out)
    with pytest.raises(B.TtsGptError) as e:
        eng.sync()
    assert e.value.code == B.E_TIMEOUT
    for t in range(30):
        got, want = out[:, 128 * t:128 * t + 128], whole[:, 128 * t:128 * t + 128]
        lost = t == tile or (kernel == 2 and t > tile and (t - tile) % 2 == 0)
        assert bool((got == mark).all()) if lost else bool(torch.equal(got, want)), t
    eng.sync()
    lg2, tk2 = _run(eng, prefix, 0)
    assert np.array_equal(lg, lg2) and np.array_equal(tk, tk2)
    for bad in ((3, 100, 0, 1000), (0, 129, 0, 1000), (1, 0, 0, 1000), (1, 100, -2, 1000), (2, 257, 0, 1000), (2, 200, 30, 1000), (2, 200, 0, 0)):
        with pytest.raises(B.TtsGptError) as e:
            eng.debug_expire_linear(*bad, out)
        assert e.value.code in (B.E_ARG, B.E_UNSUPPORTED)   # group sums have no pair kernel
    eng.destroy()


@pytest.mark.parametrize("rows", [100, 200])
@pytest.mark.parametrize("heads", [4, 6])
def test_pair_kernel_waits_for_a_late_second_cta(heads, rows):
    """The second CTA of a pair comes late to every tile: with rows of its own, with weights only (100 rows), and with neither
    (100 rows, last tile of 1152 features): nothing expires and every value is that of an undisturbed run."""
    d = 64 * heads
    cfg = C.tiny_config(d_model=d, n_head=heads, d_ff=4 * d, max_streams=1, n_pages=8)
    eng = B.TtsGpt(cfg, C.make_weights(cfg, seed=35), DEV)
    _run(eng, C.make_prefixes(cfg, [256], seed=36), 0)
    whole, late = torch.zeros((rows, 3 * d), device=DEV), torch.full((rows, 3 * d), float("nan"), device=DEV)
    torch.cuda.synchronize()
    eng.debug_expire_linear(2, rows, -1, 1000, whole)
    for _ in range(3):
        eng.debug_expire_linear(2, rows, -2, 50, late)
        eng.sync()
        assert torch.equal(late, whole)
        late.fill_(float("nan"))
        torch.cuda.synchronize()
    eng.destroy()


def test_prefill_pair_kernel_with_the_8bit_cache_and_k_ranges():
    """A model width at which the residual linears of a large pass take k-ranges, K/V rows through the staging array."""
    cfg = C.tiny_config(d_model=512, n_head=8, d_ff=2048, kv_fmt=C.KV_FP8_E4M3, max_streams=2, n_pages=40, max_context=1216, max_pos=1216)
    w = C.make_weights(cfg, seed=25)
    prefixes = C.make_prefixes(cfg, [1100, 77], seed=26)
    eng = B.TtsGpt(cfg, w, DEV)
    lg, tk = _run(eng, prefixes, 2)
    _check_e4m3(O.OracleModel(cfg, w), prefixes, lg, tk, range(2), "pair kernel, 8-bit cache")
    eng.set_option("prefill_pass_rows", 512)
    lg2, _ = _run(eng, prefixes, 2)
    assert np.max(np.abs(lg[:, 0] - lg2[:, 0])) < 4.5e-2
    assert eng.check_canaries() == 0
    eng.destroy()


@pytest.mark.parametrize("S", [1, 2, 4, 5, 75])
def test_sampled_calls_keep_their_order_of_sums(S):
    """Sampled calls have step graphs, pass sizes and (2 to 4 rows, middle batches) kernels of their own: with uniforms of
    zero they take the first of the top k, the greedy token, and greedy calls in between change nothing."""
    lens = [1030 if i == 0 else 2 + (11 * i) % 60 for i in range(S)]
    cfg = C.tiny_config(max_streams=S, n_pages=sum((x + 8 + 63) // 64 for x in lens), max_context=1152, max_pos=1152)
    w = C.make_weights(cfg, seed=27)
    model = O.OracleModel(cfg, w)
    eng = B.TtsGpt(cfg, w, DEV)
    prefixes = C.make_prefixes(cfg, lens, seed=28)
    kw = dict(top_k=4, uniforms=torch.zeros(S, device=DEV))
    lg, tk = _run(eng, prefixes, 4, **kw)
    _check(model, prefixes, lg, tk, sorted({0, S // 2, S - 1}), "sampled")
    _run(eng, prefixes, 2)
    lg2, tk2 = _run(eng, prefixes, 4, **kw)
    assert np.array_equal(lg, lg2) and np.array_equal(tk, tk2)
    assert eng.check_canaries() == 0
    eng.destroy()


ONE_UNIT_OF_MORE = {   # model, rows of a unit, prefix lengths
    "tail of 1 row": ("tiny", 1024, [1025]),
    "tail of 128 rows": ("tiny", 1024, [1100, 1000, 76]),
    "tail of 129 rows": ("tiny", 1024, [1153, 1024]),
    "two whole units": ("tiny", 1024, [2048]),
    "three units in two passes, tail of 5 rows": ("tiny", 1024, [1500, 1000, 577]),
    "many streams, heads of more than 16 rows": ("tiny", 1024, [30 + 7 * (i % 11) for i in range(40)]),
    "wide model, three units": ("wide", 896, [1900, 20, 700, 64]),
    "wide model, tail of 100 rows": ("wide", 896, [896, 996]),
    "wide model, four units": ("wide", 896, [2000, 1300]),
}


@pytest.mark.parametrize("wfmt", [C.W_BF16, C.W_INT8_PC, C.W_INT4_G128])
@pytest.mark.parametrize("form", list(ONE_UNIT_OF_MORE))
def test_sampled_passes_of_several_units_give_the_bits_of_single_units(form, wfmt):
    """A sampled prefill runs several units of rows as one pass and the last few rows apart: the same bits, tokens and
    cache (decoded from afterwards) as with passes of one unit."""
    model, unit, lens = ONE_UNIT_OF_MORE[form]
    kw = dict(wfmt=wfmt, max_streams=len(lens), n_pages=sum((x + 8 + 63) // 64 for x in lens), max_context=2048, max_pos=2048)
    if model == "wide":
        kw.update(d_model=1280, n_head=20, d_ff=5120)
    cfg = C.tiny_config(**kw)
    eng = B.TtsGpt(cfg, C.make_weights(cfg, seed=37), DEV)
    prefixes = C.make_prefixes(cfg, lens, seed=38)
    u = dict(top_k=30, uniforms=torch.rand(len(lens), generator=torch.Generator(DEV).manual_seed(3), device=DEV))
    steps = 2 if max(lens) <= 2040 else 0
    lg, tk = _run(eng, prefixes, steps, **u)
    eng.set_option("prefill_pass_rows", unit)
    lg1, tk1 = _run(eng, prefixes, steps, **u)
    assert np.array_equal(lg, lg1) and np.array_equal(tk, tk1)
    eng.destroy()


@pytest.mark.parametrize("S,d,top_k", [(11, 512, 0), (9, 1280, 0), (12, 1280, 30), (40, 1280, 0), (47, 1024, 0)])
def test_pages_asked_into_l2_change_nothing(S, d, top_k):
    """The linears of a step ask the next attention's complete pages into L2 (at these rows and widths): the same bits with and
    without, contexts with and without a complete page, more pages than the budget takes."""
    lens = [1, 63, 64, 65, 129, 700][:min(S, 6)] + [3 + (13 * i) % 200 for i in range(S - 6)]
    cfg = C.tiny_config(d_model=d, n_head=d // 64, d_ff=1536, max_streams=S, n_pages=sum((x + 8 + 63) // 64 for x in lens), max_context=768)
    eng = B.TtsGpt(cfg, C.make_weights(cfg, seed=61), DEV)
    prefixes = C.make_prefixes(cfg, lens, seed=62)
    kw = dict(top_k=top_k, uniforms=torch.full((S,), 0.3, device=DEV)) if top_k else {}
    lg, tk = _run(eng, prefixes, 3, **kw)
    eng.set_option("kv_prefetch", 0)
    lg2, tk2 = _run(eng, prefixes, 3, **kw)
    assert np.array_equal(lg, lg2) and np.array_equal(tk, tk2)
    eng.destroy()


@pytest.mark.parametrize("form", list(ONE_UNIT_OF_MORE))
def test_sampled_passes_of_several_units_over_the_8bit_cache(form):
    """The same over the 8-bit cache, whose passes decode the pages they attend over."""
    model, unit, lens = ONE_UNIT_OF_MORE[form]
    kw = dict(kv_fmt=C.KV_FP8_E4M3, max_streams=len(lens), n_pages=sum((x + 8 + 63) // 64 for x in lens), max_context=2048, max_pos=2048)
    if model == "wide":
        kw.update(d_model=1280, n_head=20, d_ff=5120)
    cfg = C.tiny_config(**kw)
    eng = B.TtsGpt(cfg, C.make_weights(cfg, seed=57), DEV)
    prefixes = C.make_prefixes(cfg, lens, seed=58)
    u = dict(top_k=30, uniforms=torch.rand(len(lens), generator=torch.Generator(DEV).manual_seed(4), device=DEV))
    steps = 2 if max(lens) <= 2040 else 0
    lg, tk = _run(eng, prefixes, steps, **u)
    eng.set_option("prefill_pass_rows", unit)
    lg1, tk1 = _run(eng, prefixes, steps, **u)
    assert np.array_equal(lg, lg1) and np.array_equal(tk, tk1)
    assert eng.check_canaries() == 0
    eng.destroy()


@pytest.mark.parametrize("wfmt,lens", [(C.W_BF16, [897]), (C.W_INT8_PC, [500, 520]), (C.W_INT4_G128, [1024]), (C.W_BF16, [640, 512, 128]),
                                       (C.W_INT8_PC, [640, 512]), (C.W_BF16, [640, 513])])
def test_prefill_passes_around_the_pair_kernels_lines(wfmt, lens):
    """897, 1020 and 1024 rows: FC2 alone on pairs, the other linears on single CTAs; 1152: all on single CTAs; 1153 and 1280: all
    on pairs."""
    cfg = C.tiny_config(wfmt=wfmt, d_model=1280, n_head=20, d_ff=5120, max_streams=len(lens), n_pages=sum(x // 64 + 2 for x in lens),
                        max_context=1088, max_pos=1088)
    w = C.make_weights(cfg, seed=59)
    model = O.OracleModel(cfg, w)
    eng = B.TtsGpt(cfg, w, DEV)
    prefixes = C.make_prefixes(cfg, lens, seed=60)
    lg, tk = _run(eng, prefixes, 1)
    _check(model, prefixes, lg, tk, range(len(lens)), "around the lines")
    assert np.array_equal(lg, _run(eng, prefixes, 1)[0])
    eng.destroy()


@pytest.mark.parametrize("S", [1, 21, 30, 40, 60, 80, 100])
def test_8bit_decode_attention_splits(S):
    """8, 6, 4, 3, 2 and 1 CTAs per (row, head) over the 8-bit cache: contexts at the edges of half pages and pages, splits
    without tokens, stale pages; against the streaming kernel on the same history, greedy and sampled order (a ticket kernel of
    five CTAs per SM up to 80 rows, of four at 100)."""
    edges = [700, 1, 30, 31, 32, 33, 62, 63, 64, 65, 95, 96, 127, 128, 161]
    lens = [edges[i % len(edges)] if i < 30 else 2 + (11 * i) % 60 for i in range(S)]
    cfg = C.tiny_config(kv_fmt=C.KV_FP8_E4M3, max_streams=S, n_pages=sum((x + 8 + 63) // 64 for x in lens), max_context=768)
    w = C.make_weights(cfg, seed=29)
    model = O.OracleModel(cfg, w)
    eng = B.TtsGpt(cfg, w, DEV)
    eng.set_option("poison_free_pages", 1)
    prefixes = C.make_prefixes(cfg, lens, seed=30)
    lg, tk = _run(eng, prefixes, 3)
    lg2, tk2 = _run(eng, prefixes, 3, top_k=4, uniforms=torch.zeros(S, device=DEV))
    streams = sorted(set(range(min(S, 15))) | {S - 1})
    _check_e4m3(model, prefixes, lg, tk, streams, "8-bit cache, greedy")
    _check_e4m3(model, prefixes, lg2, tk2, streams, "8-bit cache, sampled order")
    eng.set_option("attn_stream_min_pairs", 1)
    lg3, tk3 = _run(eng, prefixes, 3)
    for a, t in ((lg, tk), (lg2, tk2)):
        same = (t == tk3).all(axis=1)      # streams whose history is the same up to ties
        assert same.mean() > 0.9
        assert np.max(np.abs(a[same] - lg3[same])) < 4.5e-2
    assert eng.check_canaries() == 0
    eng.destroy()


@pytest.mark.parametrize("S", [5, 21, 37, 49])
def test_half_page_decode_attention(S):
    """8, 6, 4 and 3 CTAs per (row, head) over the bf16 cache: contexts at the edges of half pages and pages, splits without
    tokens, stale pages full of NaN behind every context."""
    edges = [700, 1, 30, 31, 32, 33, 62, 63, 64, 65, 95, 96, 127, 128, 161]
    lens = [edges[i % len(edges)] if i < 30 else 2 + (11 * i) % 60 for i in range(S)]
    cfg = C.tiny_config(max_streams=S, n_pages=sum((x + 8 + 63) // 64 for x in lens), max_context=768)
    w = C.make_weights(cfg, seed=31)
    model = O.OracleModel(cfg, w)
    eng = B.TtsGpt(cfg, w, DEV)
    eng.set_option("poison_free_pages", 1)
    prefixes = C.make_prefixes(cfg, lens, seed=32)
    lg, tk = _run(eng, prefixes, 4)
    _check(model, prefixes, lg, tk, sorted(set(range(min(S, 15))) | {S - 1}), "half-page attention")
    lg2, _ = _run(eng, prefixes, 4)
    assert np.array_equal(lg, lg2)
    eng.destroy()


THREADS = """
import threading, numpy as np, torch
from paper_2607_21042_b200 import binding as B, cases as C
cfgs = [C.tiny_config(wfmt=f, kv_fmt=k, max_streams=2, n_pages=48, max_context=2048, max_pos=2048) for f in (0, 1, 2) for k in (0, 1)]
weights = [C.make_weights(c, seed=41) for c in cfgs]
prefixes = [torch.from_numpy(p.view(np.int16)).to("cuda:0") for p in C.make_prefixes(cfgs[0], [1300, 70], seed=42)]
torch.cuda.synchronize()
gate, got = threading.Barrier(len(cfgs)), {}
def work(i, wait):
    torch.cuda.set_device(0)
    eng = B.TtsGpt(cfgs[i], weights[i], "cuda:0")
    lg = torch.zeros((3, 2, cfgs[i].vocab), device="cuda:0")
    tok = torch.zeros((3, 2), dtype=torch.int32, device="cuda:0")
    torch.cuda.synchronize()
    if wait:
        gate.wait(60)
    ids, _ = eng.prefill(prefixes, out_tokens=tok[0], out_logits=lg[0])
    eng.decode_steps(ids, 2, tok[1:], out_logits=lg[1:])
    eng.sync()
    got[i, wait] = lg.cpu().numpy()
ts = [threading.Thread(target=work, args=(i, True)) for i in range(len(cfgs))]
[t.start() for t in ts]
[t.join() for t in ts]
for i in range(len(cfgs)):
    work(i, False)
    assert np.array_equal(got[i, True], got[i, False]), i
print("threads ok")
"""


def test_first_calls_from_several_threads():
    """Six engines make a process's first launches at the same moment, each on a thread and stream of its own: every kernel's
    shared-memory opt-in is in place for each of them, and the results are those of one engine after the other."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", THREADS], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "threads ok" in r.stdout, r.stdout + r.stderr
