"""GPU parity of appends whose ragged ends (tokens that extend or complete an open group, tokens behind the last whole group)
go through one kernel ahead of the whole groups': every cache array bit for bit against the CPU oracle."""
import pytest
import torch

import oracle
import paper_2508_04257_b200 as kv
from paper_2508_04257_b200 import synth

from parity_util import CACHE_BUFFERS, SINK_BUFFERS, check_guards, compare_cache, configs, guard, np16

pytestmark = pytest.mark.gpu
TINY = synth.WORKLOADS["tiny"]


# chunk ends: inside the open group, on its end, with whole groups behind, with a remainder shorter and longer than the head's slots
@pytest.mark.parametrize("bits,d,group", [(2, 128, 128), (3, 128, 64), (4, 128, 64), (2, 128, 32), (3, 128, 128), (4, 64, 32), (2, 64, 64)])
@pytest.mark.parametrize("cuts", [(0.3, 0.7), (0.9, 1.0), (0.4, 3.2), (0.6, 2.95), (1.0, 2.03), (0.02, 4.0)])
def test_chunks(bits, d, group, cuts):
    ends = [max(1, int(x * group)) for x in cuts] + [5 * group + 3]
    seq = ends[-1]
    wl = TINY.scaled(bits=bits, head_dim=d, group=group, n_q_heads=6, n_kv_heads=3, batch=2, seq=seq, topk=min(seq, 9 + group // 4), pfn_n=2,
                     seed=31000 + bits * 1000 + d + group + ends[1])
    ocfg, gcfg = configs(wl)
    H = synth.make_hidden(wl, "cuda")
    K, V = synth.make_kv(wl, 0, "cuda")
    gs = guard(kv.SinkSet(gcfg), SINK_BUFFERS)
    kv.predict_sinks(gcfg, H, gs)
    gc = guard(kv.KVCache(gcfg, gs), CACHE_BUFFERS)
    bm, pos, cnt = oracle.predict_sinks(ocfg, np16(H))
    oc = oracle.Cache(ocfg, bm, pos, cnt)
    at = 0
    for end in ends:
        # [B, T, Hkv, D] storage for every other chunk
        k, v = (x[:, :, at:end] if at % 2 else x[:, :, at:end].permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for x in (K, V))
        kv.quantize_append(gcfg, gc, k, v)
        oracle.quantize_append(ocfg, oc, np16(K[:, :, at:end]), np16(V[:, :, at:end]))
        compare_cache(gc, oc, wl, f"after {end} tokens: ")
        at = end
    assert kv.read_status(gc) == 0
    check_guards(gs)
    check_guards(gc)


# schemes without token groups (static pairs, per-token keys): chunks that start between group and tile boundaries send their whole
# spans to the bulk kernel and whole tiles to the tile kernel; single tokens have a kernel of their own, on fresh and used tiles
@pytest.mark.parametrize("scheme,bits,group", [("static", 2, 128), ("static", 3, 64), ("static", 4, 64), ("static", 3, 128), ("per_token", 2, 64),
                                               ("per_token", 4, 128), ("per_token", 3, 128)])
def test_flat_chunks(scheme, bits, group):
    import test_gpu_calibrated
    import test_gpu_pertoken
    chunks = (1, 36, 2 * group + 50, 1, 2, 13, 1, group + 17, 15, 1, 1)
    wl = TINY.scaled(bits=bits, head_dim=128, group=group, n_q_heads=3, n_kv_heads=3, batch=2, seq=sum(chunks), topk=40, pfn_n=1,
                     seed=33000 + bits * 100 + group)
    (test_gpu_calibrated if scheme == "static" else test_gpu_pertoken)._both(wl, chunks=chunks)


# the whole groups' kernel of a ragged chunk starts beside the edges' kernel: its inputs, rewritten in place right before it by
# kernels of the same stream, have to be the new ones every time
@pytest.mark.parametrize("bits,group", [(3, 64), (2, 128), (4, 64)])
def test_inputs_rewritten_in_place_right_before_a_ragged_chunk(bits, group):
    T, cut, rounds = 9 * group + 11, group // 2 + 1, 8
    wl = TINY.scaled(bits=bits, head_dim=128, group=group, n_q_heads=8, n_kv_heads=8, batch=4, seq=T, topk=40, pfn_n=1, seed=32000 + bits)
    _, gcfg = configs(wl)
    sources = []
    for r in range(rounds):
        one = wl.scaled(seed=wl.seed + 10 * r)
        sources.append((synth.make_hidden(one, "cuda"), *synth.make_kv(one, 0, "cuda")))
    names = [n for n in CACHE_BUFFERS if n != "status"]

    def passes(wait):
        H, K, V = (torch.empty_like(x) for x in sources[0])
        gs = kv.SinkSet(gcfg)
        gc = kv.KVCache(gcfg, gs)
        seen = []
        torch.cuda.synchronize()
        for src in sources:
            gc.seq_len = 0
            H.copy_(src[0])
            K[:, :, :cut].copy_(src[1][:, :, :cut])
            V[:, :, :cut].copy_(src[2][:, :, :cut])
            kv.predict_sinks(gcfg, H, gs)
            wait()
            kv.quantize_append(gcfg, gc, K[:, :, :cut], V[:, :, :cut])
            wait()
            K.copy_(src[1])
            V.copy_(src[2])
            kv.predict_sinks(gcfg, H, gs)
            wait()
            kv.quantize_append(gcfg, gc, K[:, :, cut:], V[:, :, cut:])
            wait()
            seen.append([getattr(gc, n).clone() for n in names])
        assert kv.read_status(gc) == 0
        return seen

    for r, (got, ref) in enumerate(zip(passes(lambda: None), passes(torch.cuda.synchronize))):
        for n, a, b in zip(names, got, ref):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), f"{n}, round {r}"


@pytest.mark.parametrize("d,launches", [(64, 1), (128, 1)])
def test_a_chunk_without_a_whole_span_is_one_launch(d, launches):
    # 100 tokens from position 5 with G = 144: 11 up to a tile boundary, five tiles, the last nine
    cfg = kv.Config(1, 2, 2, d, 64, 2, 144, 144, 2, 1, (1,))
    g = torch.Generator("cuda").manual_seed(1)
    K, V = (torch.randn((1, 2, 105, d), device="cuda", generator=g).half() for _ in range(2))
    sinks = kv.predict_sinks(cfg, torch.randn((1, 105, 64), device="cuda", generator=g).half(), kv.SinkSet(cfg))
    params = kv.calibrate(cfg, K, V, sinks)
    cache, whole = kv.KVCache(cfg, sinks), kv.KVCache(cfg, sinks)
    kv.quantize_append_calibrated(cfg, whole, params, K, V)
    kv.quantize_append_calibrated(cfg, cache, params, K[:, :, :5], V[:, :, :5])
    before = kv.launch_count()
    kv.quantize_append_calibrated(cfg, cache, params, K[:, :, 5:], V[:, :, 5:])
    assert kv.launch_count() - before == launches
    assert torch.equal(cache.k_codes, whole.k_codes) and torch.equal(cache.v_codes, whole.v_codes)


# static appends of shapes that decode has no kernel for (codes and sink rows only): two channels a lane, four channel groups a row,
# groups longer than a row; single tokens on fresh tiles and on used ones, and chunks around tile and span boundaries
@pytest.mark.parametrize("d,bits,group", [(64, 2, 32), (64, 4, 32), (64, 2, 64), (64, 4, 64), (128, 2, 32), (128, 3, 32), (128, 4, 144), (128, 3, 144)])
def test_static_shapes_without_decode(d, bits, group):
    chunks = (1, 1, 14, 1, 20, 1, 2 * group + 35, 1, 9, 1, 1)
    wl = TINY.scaled(bits=bits, head_dim=d, group=group, n_q_heads=3, n_kv_heads=3, batch=2, seq=sum(chunks), topk=60, pfn_n=1, seed=34000 + bits + d + group)
    ocfg, gcfg = configs(wl)
    H = synth.make_hidden(wl, "cuda")
    K, V = synth.make_kv(wl, 0, "cuda")
    gs = guard(kv.SinkSet(gcfg), SINK_BUFFERS)
    kv.predict_sinks(gcfg, H, gs)
    bm, pos, cnt = oracle.predict_sinks(ocfg, np16(H))
    gp, op = kv.calibrate(gcfg, K[:, :, :90], V[:, :, :90], gs), oracle.calibrate(ocfg, np16(K[:, :, :90]), np16(V[:, :, :90]), bm)
    gc, oc = guard(kv.KVCache(gcfg, gs), CACHE_BUFFERS), oracle.Cache(ocfg, bm, pos, cnt)
    at = 0
    for n in chunks:
        k, v = K[:, :, at:at + n], V[:, :, at:at + n]
        kv.quantize_append_calibrated(gcfg, gc, gp, k, v)
        oracle.quantize_append_calibrated(ocfg, oc, op, np16(k), np16(v))
        at += n
        used, per = (at + 15) // 16 * 16 * d * bits // 8, wl.max_seq * d * bits // 8
        for name in ("k_codes", "v_codes"):
            g, o = (x.reshape(-1, per)[:, :used] for x in (getattr(gc, name).cpu().numpy(), getattr(oc, name)))
            assert g.tobytes() == o.tobytes(), f"{name} after {at} tokens"
        for name in ("sink_k", "sink_v"):
            g = getattr(gc, name).cpu().numpy().reshape(-1)
            assert g.tobytes() == getattr(oc, name).tobytes(), f"{name} after {at} tokens"
    assert kv.read_status(gc) == 0
    check_guards(gs)
    check_guards(gc)


# whole groups of 32 tokens, and of 128 at 3 bit, go to the bulk quantizer from 400 and 1200 work items (4096 elements) on; two rounds of items a warp.
# 3 bit: two items of 32 channels share the words of the high bits
def _extremes(x):
    x[:, :, :, 1] = 0.0
    x[:, :, :, 2] = -2.5
    x[:, :, :, 65] *= 300.0
    x[:, :, :, 66] = 40.0 + x[:, :, :, 66] * 0.01
    x[:, :, 5:9] = 7.0
    x[:, :, 40] *= 1e-3
    return x.clamp_(-60000, 60000)


@pytest.mark.parametrize("bits,group,batch,heads,T", [(2, 32, 8, 8, 700), (3, 32, 8, 8, 650), (4, 32, 4, 16, 671), (2, 32, 7, 3, 330), (3, 128, 4, 8, 5 * 128 + 70),
                                                      (3, 128, 8, 8, 12 * 128)])
def test_group_sizes_of_the_bulk_quantizer(bits, group, batch, heads, T):
    wl = TINY.scaled(bits=bits, head_dim=128, group=group, n_q_heads=heads, n_kv_heads=heads, batch=batch, seq=T, topk=40, pfn_n=3, seed=35000 + bits + group + T)
    ocfg, gcfg = configs(wl)
    H = synth.make_hidden(wl, "cuda")
    K, V = (_extremes(x) for x in synth.make_kv(wl, 0, "cuda"))
    gs = guard(kv.SinkSet(gcfg), SINK_BUFFERS)
    kv.predict_sinks(gcfg, H, gs)
    gc, oc = guard(kv.KVCache(gcfg, gs), CACHE_BUFFERS), oracle.Cache(ocfg, *oracle.predict_sinks(ocfg, np16(H)))
    for at, end in ((0, group + 5), (group + 5, T)):
        kv.quantize_append(gcfg, gc, K[:, :, at:end], V[:, :, at:end])
        oracle.quantize_append(ocfg, oc, np16(K[:, :, at:end]), np16(V[:, :, at:end]))
        compare_cache(gc, oc, wl, f"after {end} tokens: ")
    assert kv.read_status(gc) == 0
    check_guards(gs)
    check_guards(gc)


# the same with static pairs and per-token keys (1500 items): ragged ends in one launch ahead, with few tokens, whole tiles and both
@pytest.mark.parametrize("scheme", ["static", "per_token"])
@pytest.mark.parametrize("chunks", [(5 * 128 + 11, 3, 90), (130, 6 * 128 + 30), (16, 4 * 128 + 112, 1, 15)])
def test_flat_chunks_of_many_units(scheme, chunks):
    import test_gpu_calibrated
    import test_gpu_pertoken
    wl = TINY.scaled(bits=3, head_dim=128, group=128, n_q_heads=8, n_kv_heads=8, batch=8, seq=sum(chunks), topk=40, pfn_n=1, seed=36000 + chunks[0])
    (test_gpu_calibrated if scheme == "static" else test_gpu_pertoken)._both(wl, chunks=chunks)


# A warp of the bulk quantizer takes several items one after the other and asks for the next one while it codes the last: with inputs that
# are in L2 the next one comes soon, and must not reach the stage before every matrix of the last has left it.  84 MB of inputs, four items a warp and more,
# half of it taken again and again: the same bytes every time, which are the oracle's
@pytest.mark.parametrize("scheme,bits,group", [("static", 2, 128), ("static", 2, 64), ("static", 3, 64), ("static", 3, 128), ("static", 4, 64), ("static", 4, 128),
                                               ("per_token", 2, 64), ("per_token", 3, 128), ("dynamic", 2, 32), ("dynamic", 2, 128), ("dynamic", 3, 64), ("dynamic", 4, 128)])
def test_many_items_to_a_warp_from_cached_inputs(scheme, bits, group):
    wl = TINY.scaled(bits=bits, head_dim=128, group=group, n_q_heads=8, n_kv_heads=8, batch=10, seq=2048, topk=40, pfn_n=1, seed=37000 + 10 * group + bits)
    ocfg, gcfg = configs(wl, max_seq=2048)
    H = synth.make_hidden(wl, "cuda")
    K, V = synth.make_kv(wl, 0, "cuda")
    sinks, listed = kv.predict_sinks(gcfg, H, kv.SinkSet(gcfg)), oracle.predict_sinks(ocfg, np16(H))
    gc, oc = kv.KVCache(gcfg, sinks, per_token_keys=scheme == "per_token"), oracle.Cache(ocfg, *listed, per_token_keys=scheme == "per_token")
    if scheme == "static":
        gp, op = kv.calibrate(gcfg, K[:, :, :500], V[:, :, :500], sinks), oracle.calibrate(ocfg, np16(K[:, :, :500]), np16(V[:, :, :500]), listed[0])
        append = lambda k, v: kv.quantize_append_calibrated(gcfg, gc, gp, k, v)
        oracle.quantize_append_calibrated(ocfg, oc, op, np16(K), np16(V))
    else:
        one, ref = (kv.quantize_append, oracle.quantize_append) if scheme == "dynamic" else (kv.quantize_append_pertoken, oracle.quantize_append_pertoken)
        append = lambda k, v: one(gcfg, gc, k, v)
        ref(ocfg, oc, np16(K), np16(V))
    append(K, V)
    for name in ("k_codes", "v_codes", "sink_k", "sink_v") + (() if scheme == "static" else ("k_scale", "k_zero", "v_scale", "v_zero")):
        assert getattr(gc, name).cpu().numpy().tobytes() == getattr(oc, name).tobytes(), name
    first = [x.clone() for x in (gc.k_codes, gc.v_codes)]
    for _ in range(20):
        gc.k_codes.fill_(0xA5)
        gc.v_codes.fill_(0xA5)
        gc.seq_len = 0
        append(K[:, :, :1024], V[:, :, :1024])          # in L2 by now, which the whole of K, V and the codes would not be
        append(K[:, :, 1024:], V[:, :, 1024:])
        assert torch.equal(gc.k_codes, first[0]) and torch.equal(gc.v_codes, first[1])
    assert kv.read_status(gc) == 0
