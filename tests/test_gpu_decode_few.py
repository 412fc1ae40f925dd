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


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("rows", [1, 2, 4])
@pytest.mark.parametrize("rising", [True, False])
def test_weights_that_move_the_unit(bits, rows, rising):
    """Scores that climb (or fall) by 30 along the sequence and value rows between 2^-8 and 2^8: the reference and the unit of the weights
    move in most steps, or the first step's stays too large for the rest."""
    wl = _workload(bits, 64, 1000, rows)
    H = synth.make_hidden(wl, "cuda")
    g = torch.Generator("cuda").manual_seed(bits)
    q = torch.randn((2, 3, 128), device="cuda", generator=g).half()
    K = 0.1 * torch.randn((2, 3, 1000, 128), device="cuda", generator=g)
    along = torch.linspace(0, 30, 1000, device="cuda") * 128 ** 0.5
    K += (along if rising else along.flip(0))[:, None] * (q.float() / q.float().pow(2).sum(-1, keepdim=True))[:, :, None]
    # the other rows of a KV head climb at other rates, or fall
    q = torch.stack([q * (1 - 0.7 * r) for r in range(rows)], 2).reshape(2, 3 * rows, 128).contiguous()
    V = torch.randn((2, 3, 1000, 128), device="cuda", generator=g) * 2.0 ** (16 * torch.rand((2, 3, 1000, 1), device="cuda", generator=g) - 8)
    out, lse, (ref, ref_lse) = _both(wl, H, K.half(), V.half(), q)
    # the outputs are as large as the loudest rows near the top score: the tolerance goes with them
    assert np.abs(out - ref).max() <= (2e-3 + 1e-2) * np.abs(ref).max()
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


@pytest.mark.parametrize("bits,rows", [(2, 1), (4, 1), (2, 2), (4, 4), (3, 4)])
def test_sums_beyond_32_bits(bits, rows):
    """A query of zeros gives every token the weight 1: a warp's byte sums pass int32 unless they are carried on the way (every 2048
    tiles; 592 units leave one split, whose four warps take 2112 tiles each).  All units hold one unit's cache."""
    units, seq = 592, 4 * 2112 * 16
    one = kv.Config(1, rows, 1, 128, 512, bits, 128, seq, 2, 1, (1,))
    many = kv.Config(1, rows * units, units, 128, 512, bits, 128, seq, 2, 1, (1,))
    g = torch.Generator("cuda").manual_seed(7)
    K, V = (torch.randn((1, 1, seq, 128), device="cuda", generator=g).half() for _ in range(2))
    V += 3                                                     # most values of a row near its middle, all far from zero
    H = torch.randn((1, seq, 512), device="cuda", generator=g).half()
    sinks = kv.predict_sinks(one, H, kv.SinkSet(one))
    small = kv.KVCache(one, sinks)
    kv.quantize_append(one, small, K, V)
    big = copy.copy(small)
    big.cfg, big.sizes = many, kv.cache_sizes(many)
    for name in ("k_codes", "v_codes", "k_scale", "k_zero", "v_scale", "v_zero", "k_tail", "sink_k", "sink_v"):
        setattr(big, name, getattr(small, name).repeat(units))
    out, lse = kv.decode_attention(many, big, torch.zeros((1, rows * units, 128), device="cuda", dtype=torch.float16))
    ref, ref_lse = kv.decode_attention(one, small, torch.zeros((1, rows, 128), device="cuda", dtype=torch.float16))     # short ranges: many splits
    assert kv.read_status(small) == 0
    assert torch.equal(out, out[:, :rows].repeat(1, units, 1)) and abs(lse[0, 0].item() - np.log(seq)) < 1e-4
    # the same 32-bit arithmetic in another order: 135168 terms, each side within n * 2^-24 of the sum at worst, some 2^-20 of it in earnest
    assert (out[0, 0] - ref[0, 0]).abs().max() <= 2.0 ** -18 * ref.abs().max()
    assert (ref[0, 0] - V.float().mean((0, 1, 2))).abs().max() < 0.05
