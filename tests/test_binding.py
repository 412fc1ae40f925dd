"""The binding's own work: records of device addresses (no GPU needed: the addresses are not followed)."""
import ctypes as C
import os
import subprocess
import sys

import pytest
import torch

import paper_2508_04257_b200 as kv
from paper_2508_04257_b200 import binding, build


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


def test_a_torch_without_the_raw_stream_handle_imports():
    script = ("import torch; del torch._C._cuda_getCurrentRawStream; import paper_2508_04257_b200 as kv; "
              "print(kv.cache_sizes(kv.Config(1, 8, 8, 64, 512, 4, 32, 256, 2, 1, (1,)))['tile_bytes'])")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", script], capture_output=True, text=True, cwd=root, timeout=300)
    assert r.returncode == 0 and r.stdout.split() == ["512"], r.stderr[-2000:]


@pytest.mark.gpu
@pytest.mark.parametrize("raw", [True, False])
def test_work_goes_to_the_current_stream(raw, monkeypatch):
    if not raw:
        monkeypatch.setattr(binding, "_raw_stream", None)
    assert binding._stream() == torch.cuda.current_stream().cuda_stream
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        assert binding._stream() == side.cuda_stream != 0


@pytest.mark.parametrize("bad", ["device", pytest.param("strides", marks=pytest.mark.gpu), pytest.param("type", marks=pytest.mark.gpu)])
def test_inputs_that_the_calls_refuse(bad):
    cache = _cache()
    k = torch.zeros((1, 8, 2, 128), dtype=torch.float32 if bad == "type" else torch.float16, device="cpu" if bad == "device" else "cuda")
    k = k.transpose(2, 3) if bad == "strides" else k
    with pytest.raises(AssertionError):
        kv.quantize_append(cache.cfg, cache, k, k)
    with pytest.raises(AssertionError):
        kv.decode_attention(cache.cfg, cache, k[:, :, 0])
    with pytest.raises(AssertionError):
        kv.prefill_attention(cache.cfg, cache, k, 0)
    with pytest.raises(AssertionError):
        kv.predict_sinks(cache.cfg, k[0], cache.sinks)
    with pytest.raises(AttributeError):
        kv.decode_attention(cache.cfg, cache, None)
    assert cache.seq_len == 0


@pytest.mark.gpu
@pytest.mark.parametrize("bad", ["shape", "strides", "type"])
def test_values_unlike_the_keys_are_refused(bad):
    cache = _cache()
    k = torch.zeros((1, 8, 4, 128), dtype=torch.float16, device="cuda")
    v = {"shape": k[:, :, :2], "strides": torch.zeros((1, 4, 8, 128), dtype=torch.float16, device="cuda").transpose(1, 2), "type": k.bfloat16()}[bad]
    with pytest.raises(AssertionError):
        kv.quantize_append(cache.cfg, cache, k, v)
    with pytest.raises(AssertionError):
        kv.quantize_append_calibrated(cache.cfg, cache, kv.StaticParams(cache.cfg), k, v)
    assert cache.seq_len == 0


@pytest.mark.gpu
def test_the_calls_run_on_the_current_stream():
    """Inputs that a side stream only writes after some 20 ms: work on any other stream would read what was there before."""
    cfg = kv.Config(2, 4, 4, 128, 512, 2, 64, 256, 2, 1, (1,))
    g = torch.Generator("cuda").manual_seed(3)
    K, V = (torch.randn((2, 4, 101, 128), device="cuda", generator=g).half() for _ in range(2))
    H, q = torch.randn((2, 101, 512), device="cuda", generator=g).half(), torch.randn((2, 4, 128), device="cuda", generator=g).half()

    def run(cache, H, K, V, q):
        kv.predict_sinks(cfg, H, cache.sinks)
        kv.quantize_append(cfg, cache, K, V)
        return (*kv.decode_attention(cfg, cache, q), *kv.prefill_attention(cfg, cache, q[:, :, None], 100), cache.k_codes, cache.sinks.pos)

    want = run(kv.KVCache(cfg), H, K, V, q)
    late, cache = [torch.zeros_like(x) for x in (H, K, V, q)], kv.KVCache(cfg)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(40_000_000)
        for x, y in zip(late, (H, K, V, q)):
            x.copy_(y)
        got = run(cache, *late)
    side.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, got))


@pytest.mark.gpu
def test_calls_take_records_results_and_errors_as_ctypes_did():
    class OwnConfig(kv.Config):
        def c(self):
            return super().c()

    class OwnCache(kv.KVCache):
        def c(self):
            return super().c()

    got, refs = [], []
    for config, cache_type in ((kv.Config, kv.KVCache), (OwnConfig, OwnCache)):
        cfg = config(2, 4, 4, 128, 512, 2, 64, 256, 2, 1, (1,))
        g = torch.Generator("cuda").manual_seed(3)
        K, V = (torch.randn((2, 4, 101, 128), device="cuda", generator=g).half() for _ in range(2))
        H, q = torch.randn((2, 101, 512), device="cuda", generator=g).half(), torch.randn((2, 4, 128), device="cuda", generator=g).half()
        cache = cache_type(cfg, kv.predict_sinks(cfg, H, kv.SinkSet(cfg)))
        kv.quantize_append(cfg, cache, K, V)
        assert cache.seq_len == 101
        out, lse = torch.empty((2, 4, 128), device="cuda"), torch.empty((2, 4), device="cuda")
        work = torch.empty(cache.sizes["decode_workspace_bytes"], dtype=torch.uint8, device="cuda")
        given = kv.decode_attention(cfg, cache, q, out, lse, work)
        assert given[0] is out and given[1] is lse
        new = kv.decode_attention(cfg, cache, q)
        assert torch.equal(new[0], out) and torch.equal(new[1], lse) and new[1].shape == lse.shape
        assert kv.decode_attention(cfg, cache, q, want_lse=False)[1] is None
        whole = kv.prefill_attention(cfg, cache, q[:, :, None], 100)
        assert whole[0].shape == (2, 4, 1, 128) and whole[1].shape == (2, 4, 1)
        got.append([cache.k_codes, out, *whole])
        with pytest.raises(kv.KvsinkError):
            kv.decode_attention(config(2, 4, 4, 128, 512, 5, 64, 256, 2, 1, (1,)), cache, q, out, lse, work)      # no such code width
        refs.append([sys.getrefcount(x) for x in (cfg.batch, out, lse, work, cache.k_codes, cache.sinks)])
        for _ in range(50):
            kv.decode_attention(cfg, cache, q, out, lse, work)
            kv.quantize_append(cfg, cache, K[:, :, :0], V[:, :, :0])
        assert refs[-1][1:] == [sys.getrefcount(x) for x in (out, lse, work, cache.k_codes, cache.sinks)]
    assert all(torch.equal(a, b) for a, b in zip(*got))


@pytest.mark.gpu
def test_a_result_that_cannot_be_allocated_leaves_the_other_to_its_owner():
    cache = _cache()
    q, out = torch.zeros((1, 8, 1, 128), device="cuda").half(), torch.zeros((1, 8, 128), device="cuda")
    cfg = kv.Config(1 << 20, 1 << 20, 8, 128, 512, 2, 64, 256, 2, 1, (1,))      # an lse of four terabytes
    before = sys.getrefcount(out)
    for _ in range(5):
        with pytest.raises(torch.OutOfMemoryError):
            kv.decode_attention(cfg, cache, q, out)
        with pytest.raises(torch.OutOfMemoryError):
            kv.prefill_attention(cfg, cache, q, 0, out)
    assert sys.getrefcount(out) == before


def test_a_torch_without_cuda_builds_the_library_alone(monkeypatch, capsys):
    monkeypatch.setattr(torch.version, "cuda", None)
    monkeypatch.setattr(build.subprocess, "run", lambda *a, **k: pytest.fail("nothing to compile"))
    assert build.build_calls(force=True) is None and "without CUDA" in capsys.readouterr().out


def test_the_calls_are_built_anew_for_another_torch_or_python(monkeypatch, tmp_path):
    compiled = []

    def run(cmd, **kw):
        compiled.append([a for a in cmd if a.startswith("-DKVSINK_CALLS_ABI=")])
        (tmp_path / "_calls.so").write_bytes(b"")
        return subprocess.CompletedProcess(cmd, 0, "", "")

    monkeypatch.setattr(build, "CALLS", str(tmp_path / "_calls.so"))
    monkeypatch.setattr(build, "OBJ", str(tmp_path / "objects"))
    monkeypatch.setattr(build.subprocess, "run", run)
    for abi, builds in (("one", 1), ("one", 1), ("two", 2), ("two", 2)):
        monkeypatch.setattr(build, "calls_abi", lambda: abi)
        build.build_calls()
        assert len(compiled) == builds and compiled[-1] == [f'-DKVSINK_CALLS_ABI="{abi}"']


def test_calls_of_another_torch_are_refused(monkeypatch):
    assert binding._native().abi == build.calls_abi()
    monkeypatch.setattr(binding, "_calls", None)
    monkeypatch.setattr(build, "calls_abi", lambda: "another")
    with pytest.raises(ImportError, match="another"):
        kv.predict_sinks(None, None, None)
