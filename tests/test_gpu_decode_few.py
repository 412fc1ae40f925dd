"""Decode with few query heads per KV head (decode_few.cuh): tile pairs, lane-owned tokens, weights in fixed point."""
import copy

import numpy as np
import pytest
import torch

import oracle
import paper_2508_04257_b200 as kv
from paper_2508_04257_b200 import synth
from parity_util import assert_close, configs, np16

pytestmark = pytest.mark.gpu


def _workload(bits, group, seq, rows=1, batch=2, heads=3):
    return synth.WORKLOADS["tiny"].scaled(bits=bits, head_dim=128, group=group, n_q_heads=rows * heads, n_kv_heads=heads, batch=batch, seq=seq, topk=3, pfn_n=1)


def _both(wl, H, K, V, q):
    ocfg, gcfg = configs(wl)
    sinks = kv.predict_sinks(gcfg, H, kv.SinkSet(gcfg))
    cache = kv.KVCache(gcfg, sinks)
    kv.quantize_append(gcfg, cache, K, V)
    oc = oracle.Cache(ocfg, *oracle.predict_sinks(ocfg, np16(H)))
    oracle.quantize_append(ocfg, oc, np16(K), np16(V))
    out, lse = kv.decode_attention(gcfg, cache, q)
    assert kv.read_status(cache) == 0
    return out.cpu().numpy(), lse.cpu().numpy(), oracle.decode_attention(ocfg, oc, np16(q))


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("rows", [1, 2, 3, 4])
@pytest.mark.parametrize("group,seq", [(32, 31), (32, 352), (64, 79), (64, 1000), (128, 128), (128, 1300), (144, 577), (144, 432)])
def test_odd_lengths_and_groups(bits, rows, group, seq):
    wl = _workload(bits, group, seq, rows)
    H = synth.make_hidden(wl, "cuda")
    K, V = synth.make_kv(wl, 0, "cuda")
    out, lse, (ref, ref_lse) = _both(wl, H, K, V, synth.make_query(wl, K))
    assert_close(out, ref, "attention output")
    assert np.abs(lse - ref_lse).max() <= 2e-3 + 1e-3 * np.abs(ref_lse).max()


UNITS = 592      # as many units as the chip has slots: one split, whose four warps take a quarter of the sequence each


def _long_ranges(bits, group, K, V, q):
    """Decode of one unit's cache (K, V [seq, 128], q [rows, 128]) that all of UNITS units hold, and the oracle's result for one of them."""
    rows, seq = q.shape[0], K.shape[0]
    args = lambda units: (1, rows * units, units, 128, 512, bits, group, seq, 2, 1, (1,))
    one, many, ocfg = kv.Config(*args(1)), kv.Config(*args(UNITS)), oracle.Config(*args(1))
    K, V = K[None, None].half(), V[None, None].half()
    H = torch.randn((1, seq, 512), device="cuda", generator=torch.Generator("cuda").manual_seed(7)).half()
    small = kv.KVCache(one, kv.predict_sinks(one, H, kv.SinkSet(one)))
    kv.quantize_append(one, small, K, V)
    big = copy.copy(small)
    big.cfg, big.sizes = many, kv.cache_sizes(many)
    for name in ("k_codes", "v_codes", "k_scale", "k_zero", "v_scale", "v_zero", "k_tail", "sink_k", "sink_v"):
        setattr(big, name, getattr(small, name).repeat(UNITS))
    out, lse = kv.decode_attention(many, big, q.half().repeat(UNITS, 1)[None].contiguous())
    assert kv.read_status(small) == 0
    assert torch.equal(out, out[:, :rows].repeat(1, UNITS, 1)) and torch.equal(lse, lse[:, :rows].repeat(1, UNITS))
    oc = oracle.Cache(ocfg, *oracle.predict_sinks(ocfg, np16(H)))
    oracle.quantize_append(ocfg, oc, np16(K), np16(V))
    ref, ref_lse = oracle.decode_attention(ocfg, oc, np16(q.half())[None])
    return out[0, :rows].cpu().numpy(), lse[0, :rows].cpu().numpy(), ref[0], ref_lse[0]


def _queries(rows, g):
    """Queries of one direction, each a fifth shorter than the one before, and what a key is made of so that the first one's score is 1."""
    q = torch.randn(128, device="cuda", generator=g).half().float()
    return torch.stack([q * (1 - 0.2 * r) for r in range(rows)]).half(), q * (128 ** 0.5 / q.pow(2).sum())


def _moves(score, size, room):
    """Steps of 32 tokens in which a warp's largest weight (score in bits, value row of `size`) has outgrown its unit: the fewest of the four warps."""
    logs = (score + torch.log2(size)).reshape(4, -1, 32).amax(2).tolist()
    count = []
    for steps in logs:
        placed, n = steps[0], 0
        for w in steps:
            if w > placed + room:
                placed, n = w, n + 1
        count.append(n)
    return min(count)


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("rows", [1, 2, 4])
@pytest.mark.parametrize("scores,values", [("rise", "any"), ("rise", "fall"), ("fall", "any")])
def test_weights_that_move_the_unit(bits, rows, scores, values):
    """Scores that climb (or fall) by 300 along the sequence, over 100 bits in a warp's range of 64 steps, value rows between 2^-8 and 2^8: the
    reference and the units of the weights move in most steps, or those of the first step stay too large for the rest."""
    seq, g = 8192, torch.Generator("cuda").manual_seed(bits)
    q, key = _queries(rows, g)
    along = torch.linspace(0, 1, seq, device="cuda")
    score = 300 * (along if scores == "rise" else along.flip(0))
    size = 2.0 ** (8 - 16 * along if values == "fall" else 16 * torch.rand(seq, device="cuda", generator=g) - 8)
    room = 7 if bits == 4 and rows > 1 else 5      # bits that a weight may grow by before a move is certain
    moves = _moves(score / np.log(2), size, room)
    assert moves >= 10 if scores == "rise" else moves <= 5
    K = 0.1 * torch.randn((seq, 128), device="cuda", generator=g) + score[:, None] * key
    out, lse, ref, ref_lse = _long_ranges(bits, 64, K, torch.randn((seq, 128), device="cuda", generator=g) * size[:, None], q)
    # scores of binary32 near 433, and of sums of 128 such products: 2^-14 at worst
    assert (np.abs(out - ref).max(1) <= 2e-4 * np.abs(ref).max(1)).all()
    assert np.abs(lse - ref_lse).max() <= 1e-5 * np.abs(ref_lse).max()


# jump in nats, length of the row: the reference moves by 48 to 173 bits at once, the largest weight by up to 8 more
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("rows", [1, 2, 3, 4])
def test_one_token_far_above_the_rest(bits, rows):
    g = torch.Generator("cuda").manual_seed(11 * bits + rows)
    q, key = _queries(rows, g)
    flat = torch.randn((32768, 128), device="cuda", generator=g) + 1
    for jump, loud in ((33, 1), (45, 1), (60, 16), (60, 256), (85, 1), (85, 16), (85, 256), (120, 256)):
        K, V = torch.zeros_like(flat), flat.clone()      # equal tokens, 8192 a warp, before it
        K[-100], V[-100] = jump * key, loud * V[-100]
        out, lse, ref, ref_lse = _long_ranges(bits, 64 if bits == 2 and rows > 2 else 128, K, V, q)      # the shapes that decode_few.cuh takes
        err = np.abs(out - ref).max(1) / np.abs(ref).max(1)
        assert err.max() <= 5e-5, (jump, loud, err)
        assert np.abs(lse - ref_lse).max() <= 1e-5 * np.abs(ref_lse).max(), (jump, loud)


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("rows", [1, 2, 4])
@pytest.mark.parametrize("group", [32, 64])
def test_value_channel_groups_of_different_size(bits, rows, group):
    """The channel groups of a value row lie 2^15 apart in size: the quiet ones keep their digits."""
    g = torch.Generator("cuda").manual_seed(13 * bits + rows)
    size = torch.tensor([300.0, 0.01, 0.3, 300.0], device="cuda").repeat_interleave(32) if group == 32 else torch.tensor([300.0, 0.01], device="cuda").repeat_interleave(64)
    K, V = torch.randn((8192, 128), device="cuda", generator=g), (torch.randn((8192, 128), device="cuda", generator=g) + 1) * size
    out, lse, ref, ref_lse = _long_ranges(bits, group, K, V, 2 * torch.randn((rows, 128), device="cuda", generator=g))
    err = np.abs(out - ref).reshape(rows, -1, group).max(2) / np.abs(ref).reshape(rows, -1, group).max(2)
    # weights of 22 bits at least and scores of binary32 (below 2^5: 2^-20 each), 2048 tokens a warp; one unit for all groups: 7e-3 to 0.2
    assert err.max() <= 2e-5, err


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("rows", [1, 2, 4])
def test_a_long_tail_of_small_weights(bits, rows):
    """Each warp has one token far above 32767 others: a 2^-25th of its weight apiece (2^-20th and 2^-15th for the third and fourth row), a
    thousandth of the output together."""
    g = torch.Generator("cuda").manual_seed(17 * bits + rows)
    q, key = _queries(rows, g)
    V = torch.randn((131072, 128), device="cuda", generator=g) + 1
    for depth in (24.5, 25.2, 26, 30):
        K = torch.zeros_like(V)
        K[::32768] = depth * np.log(2) * key
        out, lse, ref, ref_lse = _long_ranges(bits, 64 if bits == 2 and rows > 2 else 128, K, V, q)
        err = np.abs(out - ref).max(1) / np.abs(ref).max(1)
        # scores of binary32 near 26 (2^-19 each), and binary32 sums of the weights: the lane that holds the large one (a 32nd, 16th or 8th of
        # a row's) loses half a digit of its sum, or a whole weight, at every small one, and so do its sums of weight * scale * zero.  Weights rounded to
        # nearest lose half of the tail, or all
        lost = np.minimum(2.0 ** (-depth * (1 - 0.2 * np.arange(rows))), 2.0 ** -24) * 32768 * {1: 1 / 32, 2: 1 / 16, 4: 1 / 8}[rows]
        assert (err <= 2e-5 + 2 * lost).all(), (depth, err, lost)


@pytest.mark.parametrize("rows,place", [(1, 28), (2, 24), (4, 24)])
def test_sums_beyond_32_bits(rows, place):
    """4 bit, all tokens weigh the same, just below the largest weight that fits, and some channels have the largest code in every token: their
    sums of bytes pass int32 unless they are carried, or added up in binary32, on the way (every 2048 tiles), and those of the top byte are
    beyond 2^29 by then.  The unit comes from a warp's first tokens, whose value rows are smaller (it puts the largest weight to 2^place).
    Codes of 2 and 3 bit add a twentieth as much: no cache is long enough."""
    tiles, weight = 4800, 1.98
    seq, g = 4 * tiles * 16, torch.Generator("cuda").manual_seed(7)
    a_tile = 16 * 15 * 16 * (int(weight * 2 ** 30) >> 24)      # tokens, code, place of the field in a byte of channels 8 to 15, top byte of the weight
    assert a_tile * (tiles - 4) > 2 ** 31 and 2 ** 31 > a_tile * 2048 > 2 ** 29
    codes = torch.randint(0, 16, (seq, 128), device="cuda", generator=g).float()
    codes[:, ::16], codes[:, 9::16] = 0, 15
    size = torch.full((4, seq // 4, 1), weight, device="cuda")
    size[:, :64] = 2.0 ** (place - 30)
    out, lse, ref, ref_lse = _long_ranges(4, 128, torch.zeros_like(codes), codes * size.reshape(seq, 1), torch.zeros((rows, 128), device="cuda"))
    # equal weights: what is left is the rounding of binary32 sums over 2400 tokens a lane
    assert np.abs(out - ref).max() <= 1e-5 * np.abs(ref).max() and np.abs(lse - np.log(seq)).max() < 1e-4
