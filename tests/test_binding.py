"""The binding's own work: records of device addresses (no GPU needed: the addresses are not followed)."""
import ctypes as C

import pytest
import torch

import paper_2508_04257_b200 as kv
from paper_2508_04257_b200 import binding


def _cache():
    return kv.KVCache(kv.Config(1, 8, 8, 128, 512, 2, 64, 256, 2, 1, (1,)), device="cpu")


@pytest.mark.parametrize("dropped", [("k_tail",), ("k_scale", "k_zero", "v_scale", "v_zero", "k_tail"), ("sink_k", "sink_v")])
def test_buffers_that_a_scheme_does_not_use_may_be_dropped(dropped):
    cache = _cache()
    whole = cache.c()
    for name in dropped:
        setattr(cache, name, None)
    record = cache.c()
    for name, _ in binding._Cache._fields_:
        assert getattr(record, name) == (None if name in dropped else getattr(whole, name)), name


def test_a_buffer_that_every_scheme_needs_is_refused_by_the_library():
    cache = _cache()
    cache.k_codes = None
    record = cache.c()
    assert binding.lib().kvsink_quantize_append(C.byref(cache.cfg.c()), C.byref(record), 16, 16, 1, 1024, 128, 128, None) == -1


@pytest.mark.gpu
def test_static_parameters_without_the_arrays_they_do_not_use():
    cfg = kv.Config(2, 4, 4, 128, 512, 2, 64, 256, 2, 1, (1,))
    g = torch.Generator("cuda").manual_seed(3)
    K, V = (torch.randn((2, 4, 101, 128), device="cuda", generator=g).half() for _ in range(2))
    H = torch.randn((2, 101, 512), device="cuda", generator=g).half()
    q = torch.randn((2, 4, 128), device="cuda", generator=g).half()
    sinks = kv.predict_sinks(cfg, H, kv.SinkSet(cfg))
    params = kv.calibrate(cfg, K, V, sinks)
    got = []
    for dropped in ((), ("k_scale", "k_zero", "v_scale", "v_zero", "k_tail")):
        cache = kv.KVCache(cfg, sinks)
        for name in dropped:
            setattr(cache, name, None)
        kv.quantize_append_calibrated(cfg, cache, params, K, V)
        got.append((*kv.decode_attention_calibrated(cfg, cache, params, q), cache.k_codes, cache.v_codes))
    assert all(torch.equal(a, b) for a, b in zip(*got))
