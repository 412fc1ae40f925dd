"""GPU parity of prompt attention on the 256-row tensor-core blocks (head size 128, many rows) against the CPU oracle:
|gpu - oracle| <= 2e-3 + 1e-2 |oracle| for every query row, at the edges of row tiles, steps and key groups."""
import numpy as np
import pytest
import torch

import oracle
import paper_2508_04257_b200 as kv
from paper_2508_04257_b200 import synth

from parity_util import assert_close, configs, np16

pytestmark = pytest.mark.gpu
TINY = synth.WORKLOADS["tiny"]


def _check(wl, T, pos0, shape_keys=None, shape_values=None, strided=False, rows=256):
    ocfg, gcfg = configs(wl)
    H = synth.make_hidden(wl, "cuda")
    K, V = synth.make_kv(wl, 0, "cuda")
    if shape_keys:
        shape_keys(K)
    if shape_values:
        shape_values(V)
    gs = kv.SinkSet(gcfg)
    kv.predict_sinks(gcfg, H, gs)
    bm, pos, cnt = oracle.predict_sinks(ocfg, np16(H))
    gc, oc = kv.KVCache(gcfg, gs), oracle.Cache(ocfg, bm, pos, cnt)
    kv.quantize_append(gcfg, gc, K, V)
    oracle.quantize_append(ocfg, oc, np16(K), np16(V))
    g = torch.Generator("cuda").manual_seed(wl.seed + T)
    q = torch.randn((wl.batch, wl.n_q_heads, T, wl.head_dim), device="cuda", generator=g).half()
    if strided:     # [B, T, Hq, D] storage
        q = q.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    assert kv.prefill_rows(gcfg, T) == rows
    out, lse = kv.prefill_attention(gcfg, gc, q, pos0)
    ref, ref_lse = oracle.prefill_attention(ocfg, oc, np16(q), pos0)
    torch.cuda.synchronize()
    assert kv.read_status(gc) == 0
    # an output is a mean of values with weights that carry 22 bits: its error goes with the largest value
    top = float(V.abs().max())
    assert_close(out.cpu().numpy(), ref, "prompt attention", atol=2e-3 * max(1.0, top / 6.0))
    assert np.abs(lse.cpu().numpy() - ref_lse).max() <= 2e-3 + 1e-3 * np.abs(ref_lse).max()
    return [np.linalg.norm(x.cpu().numpy() - r) / np.linalg.norm(r) for x, r in ((out, ref), (lse, ref_lse))]


# rows of a unit: 64, 8 x 63, 8 x 129 (five blocks), 4 x 257, 3 x 171 = 513, 513; sequence ends inside a step, a tile, a group
@pytest.mark.parametrize("bits,group,hq,hkv,batch,T,pos0", [
    (2, 128, 16, 16, 8, 64, 0), (4, 64, 64, 8, 8, 63, 70), (3, 64, 32, 4, 8, 129, 0), (2, 32, 16, 4, 2, 257, 0),
    (4, 144, 12, 4, 4, 171, 29), (2, 128, 4, 4, 4, 513, 0), (3, 128, 8, 8, 16, 256, 1), (4, 32, 8, 8, 8, 130, 190)])
@pytest.mark.parametrize("topk", [3, 90])
def test_tiles(bits, group, hq, hkv, batch, T, pos0, topk):
    wl = TINY.scaled(bits=bits, head_dim=128, group=group, n_q_heads=hq, n_kv_heads=hkv, batch=batch, seq=pos0 + T, topk=min(topk, pos0 + T),
                     pfn_n=2, seed=21000 + bits * 100 + group + T + topk)
    _check(wl, T, pos0, strided=T % 2 == 1)


def _wide(K):
    n = K.shape[2]
    K[:, :, :, 3] = 2.5
    K[:, :, :, 4] = 0.0
    K[:, :, :, 6] *= 300.0
    K[:, :, :, 70] *= 1e-3
    K[:, :, :, 8] = 300.0 + torch.arange(n, device="cuda").half() * 0.25
    K[:, :, :, 100] = -40.0 + torch.randn(n, device="cuda", generator=torch.Generator("cuda").manual_seed(5)).half() * 0.01


def _far(x):           # narrow ranges far from zero: zero points of some ten thousands
    x[:, :, :, ::3] = 40.0 + x[:, :, :, ::3] * 0.02
    x[:, :, :, 1::3] = -500.0 + x[:, :, :, 1::3] * 0.3


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("keys,values", [(_wide, None), (None, _far), (_far, _far), (lambda K: K.mul_(1e-3), lambda V: V.mul_(1e-4)),
                                         (lambda K: K.mul_(8.0), lambda V: V.mul_(8000.0).clamp_(-60000, 60000))])
def test_ranges(bits, keys, values):
    wl = TINY.scaled(bits=bits, head_dim=128, group=32, n_q_heads=16, n_kv_heads=4, batch=2, seq=300, topk=6, pfn_n=1, seed=22000 + bits)
    _check(wl, 300, 0, keys, values)


def test_every_token_a_sink():
    wl = TINY.scaled(bits=2, head_dim=128, group=64, n_q_heads=16, n_kv_heads=4, batch=2, seq=270, topk=270, pfn_n=0, seed=23000)
    _check(wl, 270, 0)


# one step holds all sinks: up to eight of its rows are left in shared memory by the warps that look at them first, the others are not
@pytest.mark.parametrize("bits,topk", [(2, 7), (3, 8), (4, 9), (2, 17)])
def test_sink_rows_of_one_step(bits, topk):
    wl = TINY.scaled(bits=bits, head_dim=128, group=32, n_q_heads=32, n_kv_heads=16, batch=4, seq=64, topk=topk, pfn_n=0, seed=23100 + topk)
    _check(wl, 64, 0)


def _prompt(wl):
    """A cache that holds a whole prompt, and queries for all of it."""
    _, gcfg = configs(wl)
    gs = kv.predict_sinks(gcfg, synth.make_hidden(wl, "cuda"), kv.SinkSet(gcfg))
    K, V = synth.make_kv(wl, 0, "cuda")
    gc = kv.KVCache(gcfg, gs)
    kv.quantize_append(gcfg, gc, K, V)
    q = torch.randn((wl.batch, wl.n_q_heads, wl.seq, wl.head_dim), device="cuda", generator=torch.Generator("cuda").manual_seed(wl.seed)).half()
    return gcfg, gc, q


# Keys, values and weights are carried as fp16 pairs (22 bits).  Without the second half of one of them a factor keeps 11 bits, which
# moves every weight or value by up to 2^-12 of itself, some 1.5e-4 in the mean, and the outputs, whose terms carry random signs, as much
# (a numpy model of each of the three gives 1.6e-4 to 2.1e-4).  Sums in 32 bits over a few hundred terms stay below 1e-5
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("hq,hkv,T,pos0", [(16, 4, 400, 0), (16, 16, 300, 77)])
def test_precision(bits, hq, hkv, T, pos0):
    wl = TINY.scaled(bits=bits, head_dim=128, group=64, n_q_heads=hq, n_kv_heads=hkv, batch=2, seq=pos0 + T, topk=6, pfn_n=1, seed=27000 + bits)
    out, lse = _check(wl, T, pos0)
    assert out <= 3e-5 and lse <= 1e-6, (out, lse)


# queries whose last one is not the cache's last token: a step's and a group's tokens behind them are masked, the open group among them
@pytest.mark.parametrize("bits,group,behind", [(2, 128, 1), (3, 64, 63), (4, 64, 200), (2, 32, 500)])
def test_chunk_that_ends_before_the_cache(bits, group, behind):
    wl = TINY.scaled(bits=bits, head_dim=128, group=group, n_q_heads=16, n_kv_heads=8, batch=4, seq=310 + behind, topk=40, pfn_n=1, seed=28000 + bits + behind)
    _check(wl, 210, 100)


def test_without_the_log_sum():
    wl = TINY.scaled(bits=4, head_dim=128, group=64, n_q_heads=16, n_kv_heads=8, batch=2, seq=257, topk=6, pfn_n=1, seed=28500)
    gcfg, gc, q = _prompt(wl)
    assert kv.prefill_rows(gcfg, wl.seq) == 256
    out, lse = kv.prefill_attention(gcfg, gc, q, 0, want_lse=False)
    assert lse is None and torch.equal(out, kv.prefill_attention(gcfg, gc, q, 0)[0])


# a mask bit without an entry in the position list: the token has no row anywhere, so it takes no part, as on the eight-row blocks
@pytest.mark.parametrize("bits", [2, 4])
def test_mask_bit_without_a_list_entry(bits):
    wl = TINY.scaled(bits=bits, head_dim=128, group=64, n_q_heads=16, n_kv_heads=8, batch=2, seq=300, topk=6, pfn_n=1, seed=29000 + bits)
    gcfg, gc, q = _prompt(wl)
    listed = set(gc.sinks.pos.cpu().tolist())
    extra = [t for t in (2, 64, 100, 130, 131, 255, 290) if t not in listed]
    words = gc.sinks.bitmask.view(wl.batch, -1)
    for t in extra:
        words[:, t // 32] |= (1 << t % 32) - (1 << 32 if t % 32 == 31 else 0)
    assert kv.prefill_rows(gcfg, 300) == 256 and kv.prefill_rows(gcfg, 12) == 8
    out, lse = kv.prefill_attention(gcfg, gc, q, 0)
    for t in range(0, 300, 12):
        small, small_lse = kv.prefill_attention(gcfg, gc, q[:, :, t:t + 12], t)
        assert_close(out[:, :, t:t + 12].cpu().numpy(), small.cpu().numpy(), f"queries {t}")
        assert (lse[:, :, t:t + 12] - small_lse).abs().max() <= 2e-3 + 1e-3 * small_lse.abs().max()


def _same_every_time(gcfg, gc, q, pos0, times):
    first = kv.prefill_attention(gcfg, gc, q, pos0)
    for _ in range(times):
        out, lse = (torch.full_like(x, float("nan")) for x in first)
        kv.prefill_attention(gcfg, gc, q, pos0, out=out, lse=lse)
        assert torch.equal(out, first[0]) and torch.equal(lse, first[1])
    assert kv.read_status(gc) == 0


# one query head per KV head: the second row tile of a block has two steps more than the first, which ends while the other's products go on
@pytest.mark.parametrize("bits,T", [(2, 700), (3, 333), (4, 512)])
def test_a_tile_that_ends_before_the_other(bits, T):
    wl = TINY.scaled(bits=bits, head_dim=128, group=64, n_q_heads=16, n_kv_heads=16, batch=2, seq=T, topk=5, pfn_n=1, seed=24000 + bits)
    _check(wl, T, 0)
    _same_every_time(*_prompt(wl), 0, times=20)


# long streams of steps: the weights of a step make room for the scores of a later one many times over
@pytest.mark.parametrize("bits,hq,hkv,batch", [(2, 32, 8, 2), (3, 8, 8, 4), (4, 64, 8, 1)])
def test_many_steps_over_the_same_score_buffers(bits, hq, hkv, batch):
    wl = TINY.scaled(bits=bits, head_dim=128, group=128, n_q_heads=hq, n_kv_heads=hkv, batch=batch, seq=3000, topk=30, pfn_n=1, seed=24100 + bits)
    gcfg, gc, q = _prompt(wl)
    assert kv.prefill_rows(gcfg, 900) == 256
    _same_every_time(gcfg, gc, q[:, :, -900:], 2100, times=10)


# a sink token's row may hold infinities and NaN (it is kept as it came): queries before it must not see them
@pytest.mark.parametrize("bits,topk", [(2, 6), (3, 6), (4, 90)])
def test_sink_rows_that_are_not_finite_stay_hidden_from_queries_before_them(bits, topk):
    wl = TINY.scaled(bits=bits, head_dim=128, group=32, n_q_heads=16, n_kv_heads=4, batch=2, seq=300, topk=topk, pfn_n=1, seed=25000 + bits)
    ocfg, gcfg = configs(wl)
    H = synth.make_hidden(wl, "cuda")
    K, V = synth.make_kv(wl, 0, "cuda")
    bm, pos, cnt = oracle.predict_sinks(ocfg, np16(H))
    gc, oc = kv.KVCache(gcfg, kv.predict_sinks(gcfg, H, kv.SinkSet(gcfg))), oracle.Cache(ocfg, bm, pos, cnt)
    kv.quantize_append(gcfg, gc, K, V)
    oracle.quantize_append(ocfg, oc, np16(K), np16(V))
    slot = [int(cnt[b]) // 2 for b in range(2)]
    at = [int(pos[b, s]) for b, s in enumerate(slot)]
    assert all(0 < t < 290 for t in at)
    for b, s in enumerate(slot):          # [sequence, KV head, slot, channel]
        for cache in (gc, oc):
            k, v = (x.view(2, 4, -1, 128) if cache is gc else x.view(np.float16).reshape(2, 4, -1, 128) for x in (cache.sink_k, cache.sink_v))
            v[b, 0, s, 5], v[b, 1, s, 7], v[b, 1, s, 127], v[b, 2, s, 0], k[b, 3, s, 64] = np.inf, -np.inf, np.inf, np.nan, np.inf
    q = torch.randn((2, 16, 300, 128), device="cuda", generator=torch.Generator("cuda").manual_seed(wl.seed)).half()
    out, lse = (x.cpu().numpy() for x in kv.prefill_attention(gcfg, gc, q, 0))
    ref, ref_lse = oracle.prefill_attention(ocfg, oc, np16(q), 0)
    assert kv.read_status(gc) == 0
    for b, t in enumerate(at):
        out[b, 12:, t:], lse[b, 12:, t:], ref[b, 12:, t:], ref_lse[b, 12:, t:] = 0, 0, 0, 0      # queries that see the infinite key
    assert np.array_equal(np.isfinite(out), np.isfinite(ref))
    for value in (np.inf, -np.inf):
        assert np.array_equal(out == value, ref == value)
    fine = np.isfinite(ref)
    assert_close(out[fine], ref[fine], "prompt attention")
    assert np.abs(lse - ref_lse).max() <= 2e-3 + 1e-3 * np.abs(ref_lse).max()


# few rows a unit, on the side of the line that the tensor-core blocks take, with one row tile and with two; and just on the other side of it
@pytest.mark.parametrize("bits,group,hq,hkv,batch,T,pos0,rows", [
    (2, 128, 8, 8, 8, 128, 0, 256), (2, 64, 32, 8, 5, 52, 200, 256), (4, 64, 8, 8, 5, 104, 30, 256), (4, 32, 16, 8, 4, 64, 64, 256), (3, 64, 8, 8, 5, 57, 5, 256), (3, 128, 32, 8, 5, 15, 120, 256),
    (2, 128, 8, 8, 1, 1024, 0, 256), (2, 128, 8, 8, 8, 120, 0, 8), (4, 64, 8, 8, 5, 96, 0, 8), (3, 64, 8, 8, 5, 56, 5, 8)])
def test_few_rows_on_both_sides_of_the_line(bits, group, hq, hkv, batch, T, pos0, rows):
    wl = TINY.scaled(bits=bits, head_dim=128, group=group, n_q_heads=hq, n_kv_heads=hkv, batch=batch, seq=pos0 + T, topk=4, pfn_n=1, seed=32000 + bits * 100 + T)
    _check(wl, T, pos0, strided=T % 2 == 1, rows=rows)


# several row blocks to a block of the grid, which takes them one after the other: the last ones are their units' first rows, 44 with one row tile, 4, 256
@pytest.mark.parametrize("bits,group,hq,hkv,batch,T,pos0", [(2, 128, 16, 16, 12, 300, 0), (4, 64, 8, 4, 40, 130, 50), (3, 32, 4, 4, 60, 512, 0)])
def test_several_row_blocks_to_a_block(bits, group, hq, hkv, batch, T, pos0):
    wl = TINY.scaled(bits=bits, head_dim=128, group=group, n_q_heads=hq, n_kv_heads=hkv, batch=batch, seq=pos0 + T, topk=5, pfn_n=1, seed=30000 + bits)
    _check(wl, T, pos0)
    _same_every_time(*_prompt(wl)[:2], _queries(wl, T), pos0, times=3)


def _queries(wl, T):
    return torch.randn((wl.batch, wl.n_q_heads, T, wl.head_dim), device="cuda", generator=torch.Generator("cuda").manual_seed(wl.seed)).half()


# more row blocks than the lists of 148 blocks hold (95 each): twice as many blocks take them in turn, half of which begin when the others have ended.  All of
# them against the eight-row blocks, which eight queries a unit go to, and some sequences, whose 32 heads lie in blocks next to one another, against the oracle
def test_more_row_blocks_than_the_grid_takes():
    wl = TINY.scaled(bits=2, head_dim=128, group=64, n_q_heads=32, n_kv_heads=32, batch=450, seq=72, topk=2, pfn_n=1, seed=31000)
    gcfg, gc, q = _prompt(wl)
    assert wl.batch * 32 > 148 * 95 and kv.prefill_rows(gcfg, 72) == 256 and kv.prefill_rows(gcfg, 8) == 8
    out, lse = kv.prefill_attention(gcfg, gc, q, 0)
    for t in range(0, 72, 8):
        small, small_lse = kv.prefill_attention(gcfg, gc, q[:, :, t:t + 8], t)
        assert (out[:, :, t:t + 8] - small).abs().max() <= 2e-3 + 1e-2 * small.abs().max()
        assert (lse[:, :, t:t + 8] - small_lse).abs().max() <= 2e-3 + 1e-3 * small_lse.abs().max()
    assert kv.read_status(gc) == 0
    H, (K, V), (ocfg, _) = synth.make_hidden(wl, "cuda"), synth.make_kv(wl, 0, "cuda"), configs(wl.scaled(batch=1))
    for b in (0, 3, 5, 222, 438, 439, 449):
        oc = oracle.Cache(ocfg, *oracle.predict_sinks(ocfg, np16(H[b:b + 1])))
        oracle.quantize_append(ocfg, oc, np16(K[b:b + 1]), np16(V[b:b + 1]))
        ref, ref_lse = oracle.prefill_attention(ocfg, oc, np16(q[b:b + 1]), 0)
        error = lambda x, r: np.linalg.norm(x[b].cpu().numpy() - r[0]) / np.linalg.norm(r)
        assert error(out, ref) <= 3e-5 and error(lse, ref_lse) <= 1e-6, b          # the bounds of test_precision


def _many_items(wl, T, pos0, looked_at, shape_keys=None, shape_values=None, strided=False, sink_values=None):
    """More row blocks than SMs, so that blocks of the grid take several; the oracle has the sequences `looked_at`.  sink_values changes [B, Hkv, slot, D]."""
    (ocfg, _), gcfg = configs(wl.scaled(batch=1)), configs(wl)[1]
    g = torch.Generator("cuda").manual_seed(wl.seed)
    H = torch.randn((wl.batch, wl.seq, wl.hidden), device="cuda", generator=g).half()
    K, V = (torch.randn((wl.batch, wl.n_kv_heads, wl.seq, 128), device="cuda", generator=g, dtype=torch.float16) for _ in range(2))
    if shape_keys:
        shape_keys(K)
    if shape_values:
        shape_values(V)
    gc = kv.KVCache(gcfg, kv.predict_sinks(gcfg, H, kv.SinkSet(gcfg)))
    kv.quantize_append(gcfg, gc, K, V)
    if sink_values:
        sink_values(gc.sink_v.view(wl.batch, wl.n_kv_heads, -1, 128))
    q = torch.randn((wl.batch, wl.n_q_heads, T, 128), device="cuda", generator=g).half()
    if strided:
        q = q.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    assert kv.prefill_rows(gcfg, T) == 256 and wl.batch * wl.n_kv_heads * -(-T * wl.n_q_heads // wl.n_kv_heads // 256) > 148
    out, lse = (x.cpu().numpy() for x in kv.prefill_attention(gcfg, gc, q, pos0))
    assert kv.read_status(gc) == 0
    top, rows = float(V.abs().max()), gc.sink_v.cpu().numpy().view(np.uint16).reshape(wl.batch, -1)
    for b in looked_at:
        oc = oracle.Cache(ocfg, *oracle.predict_sinks(ocfg, np16(H[b:b + 1])))
        oracle.quantize_append(ocfg, oc, np16(K[b:b + 1]), np16(V[b:b + 1]))
        oc.sink_v[...] = rows[b].reshape(oc.sink_v.shape)
        ref, ref_lse = (x[0] for x in oracle.prefill_attention(ocfg, oc, np16(q[b:b + 1]), pos0))
        fine = np.isfinite(ref)
        assert np.array_equal(np.isfinite(out[b]), fine) and all(np.array_equal(out[b] == x, ref == x) for x in (np.inf, -np.inf)), f"sequence {b}"
        assert_close(out[b][fine], ref[fine], f"sequence {b}", atol=2e-3 * max(1.0, top / 6.0))
        assert np.abs(lse[b] - ref_lse).max() <= 2e-3 + 1e-3 * np.abs(ref_lse).max()
    return out


# 160 row blocks of one unit each: twelve blocks of the grid take two, and units 140 and 155 (heads 4 of sequence 17, 3 of sequence 19) share one.
# The walk over thousands of sinks for the values that the products leave out must not stand between a block's items, whose waits are bounded
@pytest.mark.parametrize("b,h", [(17, 4), (19, 3)])
@pytest.mark.parametrize("bits", [2, 4])
def test_values_that_are_not_finite_in_one_unit_among_thousands_of_sinks(bits, b, h):
    wl = TINY.scaled(bits=bits, head_dim=128, group=64, n_q_heads=8, n_kv_heads=8, batch=20, seq=4600, topk=4096, pfn_n=1, seed=38000 + bits)

    def sink_values(v):                            # [sequence, KV head, slot, channel]; the last slots are tokens among the queries'
        v[b, h, 7, 5], v[b, h, 2000, 5], v[b, h, 1999, 80], v[b, h, 4090, 64] = float("inf"), float("inf"), float("nan"), float("-inf")
        v[b, h, 4000, 127], v[b, h, 4080, 127] = float("inf"), float("-inf")

    out = _many_items(wl, 256, 4344, (0, 17, 19), sink_values=sink_values)
    wrong = ~np.isfinite(out)
    assert wrong[b, h].any() and wrong.sum() == wrong[b, h].sum()


# rows of a unit: 400 = 256 + 144 and 280 = 256 + 24 (one row tile), 130
@pytest.mark.parametrize("bits,group,T,pos0,keys,values,strided", [
    (2, 64, 100, 70, _far, _far, True), (3, 32, 100, 70, _wide, _far, False), (4, 128, 70, 131, _far, None, True), (3, 64, 70, 0, None, _far, True)])
def test_ranges_and_strides_with_several_row_blocks_to_a_block(bits, group, T, pos0, keys, values, strided):
    wl = TINY.scaled(bits=bits, head_dim=128, group=group, n_q_heads=32, n_kv_heads=8, batch=12, seq=pos0 + T, topk=20, pfn_n=1, seed=39000 + bits + T)
    _many_items(wl, T, pos0, (0, 5, 11), keys, values, strided)


# mask bits without an entry in the position list, over several row blocks to a block: against the eight-row blocks, as with one
@pytest.mark.parametrize("bits", [2, 3, 4])
def test_mask_bits_without_a_list_entry_with_several_row_blocks_to_a_block(bits):
    wl = TINY.scaled(bits=bits, head_dim=128, group=64, n_q_heads=32, n_kv_heads=8, batch=12, seq=80, topk=6, pfn_n=1, seed=39500 + bits)
    gcfg, gc, q = _prompt(wl)
    listed = set(gc.sinks.pos.cpu().tolist())
    words = gc.sinks.bitmask.view(wl.batch, -1)
    for t in (t for t in (2, 31, 40, 63, 64, 79) if t not in listed):
        words[:, t // 32] |= (1 << t % 32) - (1 << 32 if t % 32 == 31 else 0)
    assert kv.prefill_rows(gcfg, 80) == 256 and kv.prefill_rows(gcfg, 4) == 8
    out, lse = kv.prefill_attention(gcfg, gc, q, 0)
    for t in range(0, 80, 4):
        small, small_lse = kv.prefill_attention(gcfg, gc, q[:, :, t:t + 4], t)
        assert_close(out[:, :, t:t + 4].cpu().numpy(), small.cpu().numpy(), f"queries {t}")
        assert (lse[:, :, t:t + 4] - small_lse).abs().max() <= 2e-3 + 1e-3 * small_lse.abs().max()


# a mask bit without an entry ahead of thousands that have one: every sink token behind it has to be looked up, within the other warps' bounded waits
def test_mask_bit_without_a_list_entry_ahead_of_thousands_of_sinks():
    wl = TINY.scaled(bits=2, head_dim=128, group=64, n_q_heads=8, n_kv_heads=8, batch=2, seq=4300, topk=4096, pfn_n=0, seed=39900)
    _, gcfg = configs(wl)
    g = torch.Generator("cuda").manual_seed(wl.seed)
    H = torch.randn((2, 4300, wl.hidden), device="cuda", generator=g).half()
    H[:, :70] = 0                     # none of the sinks
    K, V = (torch.randn((2, 8, 4300, 128), device="cuda", generator=g, dtype=torch.float16) for _ in range(2))
    gc = kv.KVCache(gcfg, kv.predict_sinks(gcfg, H, kv.SinkSet(gcfg)))
    kv.quantize_append(gcfg, gc, K, V)
    gc.sinks.bitmask.view(2, -1)[:, 0] |= 1 << 3
    gc.sinks.bitmask.view(2, -1)[:, 2] |= 1 << 1
    q = torch.randn((2, 8, 1000, 128), device="cuda", generator=g).half()
    assert kv.prefill_rows(gcfg, 1000) == 256 and kv.prefill_rows(gcfg, 40) == 8
    out, lse = kv.prefill_attention(gcfg, gc, q, 3300)
    for t in range(0, 1000, 200):
        small, small_lse = kv.prefill_attention(gcfg, gc, q[:, :, t:t + 40], 3300 + t)
        assert_close(out[:, :, t:t + 40].cpu().numpy(), small.cpu().numpy(), f"queries {t}")
        assert (lse[:, :, t:t + 40] - small_lse).abs().max() <= 2e-3 + 1e-3 * small_lse.abs().max()


# Just above the line with some thousands of cached tokens and values in narrow ranges far from zero: sums in TMEM lose up to one unit in the 24th place of what
# they stand at, in one direction, at each of a step's twelve products of values, so 64 steps may lose 12 * 64 * 2^-24 = 4.6e-5 of an output
@pytest.mark.parametrize("bits,T", [(2, 208), (3, 57), (4, 104)])
def test_values_far_from_zero_behind_a_long_past(bits, T):
    wl = TINY.scaled(bits=bits, head_dim=128, group=64, n_q_heads=8, n_kv_heads=8, batch=5, seq=4096, topk=8, pfn_n=1, seed=40000 + bits)
    out, lse = _check(wl, T, 4096 - T, None, _far)
    assert out <= 1e-4 and lse <= 1e-6, (out, lse)
