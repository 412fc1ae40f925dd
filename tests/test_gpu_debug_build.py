"""The debug build of the library (-DKVSINK_DEBUG: index checks that raise a status bit and skip the access, never a
trap) runs the same parity cases as the release build with a clean status word.  It runs in a process of its own because
a process binds one build of the library."""
import os
import subprocess
import sys

import pytest

from paper_2508_04257_b200 import build as kv_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import sys
sys.path.insert(0, sys.argv[1]); sys.path.insert(0, sys.argv[1] + "/tests")
import torch
import paper_2508_04257_b200 as kv
from paper_2508_04257_b200 import binding, synth
from parity_util import run_both
assert binding.lib()._name.endswith("libkvsink_debug.so")
TINY = synth.WORKLOADS["tiny"]
run_both(TINY, appends=3)
for bits, group, hq, hkv in ((2, 128, 4, 4), (3, 64, 8, 2), (4, 64, 16, 2), (2, 64, 6, 2)):
    wl = TINY.scaled(bits=bits, head_dim=128, group=group, n_q_heads=hq, n_kv_heads=hkv, batch=2, seq=3 * group + 37, topk=5, pfn_n=2, seed=99 + bits)
    r = run_both(wl, appends=2)          # asserts parity and a zero status word
print("debug build ok")
"""


@pytest.mark.gpu
def test_debug_build_runs_the_path_with_a_clean_status_word():
    if not os.path.exists(kv_build.DEBUG_LIB):
        pytest.skip("libkvsink_debug.so has not been built (python -m paper_2508_04257_b200.build --debug)")
    env = dict(os.environ, KVSINK_LIB=kv_build.DEBUG_LIB)
    r = subprocess.run([sys.executable, "-c", SCRIPT, ROOT], capture_output=True, text=True, env=env, timeout=600)
    assert r.returncode == 0 and "debug build ok" in r.stdout, r.stdout[-1500:] + r.stderr[-3000:]


PROMPTS = r"""
import sys
sys.path.insert(0, sys.argv[1]); sys.path.insert(0, sys.argv[1] + "/tests")
from paper_2508_04257_b200 import synth
from test_gpu_prompt_tiles import _check, _far
TINY = synth.WORKLOADS["tiny"]
for bits, group, hq, hkv, batch, T, pos0, topk in ((2, 128, 16, 16, 8, 64, 0, 3), (4, 144, 12, 4, 4, 171, 29, 90), (3, 64, 32, 4, 8, 129, 0, 90),
                                                   (4, 32, 8, 8, 8, 130, 190, 3)):
    wl = TINY.scaled(bits=bits, head_dim=128, group=group, n_q_heads=hq, n_kv_heads=hkv, batch=batch, seq=pos0 + T, topk=min(topk, pos0 + T), pfn_n=2,
                     seed=26000 + bits)
    _check(wl, T, pos0)                  # asserts parity and a zero status word
_check(TINY.scaled(bits=2, head_dim=128, group=32, n_q_heads=16, n_kv_heads=4, batch=2, seq=300, topk=6, pfn_n=1, seed=26100), 300, 0, _far, _far)
# several work items to a block, their order among what is checked: the last ones with one row tile, with two
for bits, group, hq, hkv, batch, T, pos0 in ((2, 128, 16, 16, 12, 300, 0), (3, 64, 32, 8, 12, 100, 70), (4, 64, 8, 4, 40, 130, 50)):
    wl = TINY.scaled(bits=bits, head_dim=128, group=group, n_q_heads=hq, n_kv_heads=hkv, batch=batch, seq=pos0 + T, topk=5, pfn_n=1, seed=26200 + bits)
    _check(wl, T, pos0)
print("debug prompts ok")
"""


@pytest.mark.gpu
def test_prompts_of_many_rows_run_with_index_checks_and_a_clean_status_word():
    if not os.path.exists(kv_build.DEBUG_LIB):
        pytest.skip("libkvsink_debug.so has not been built (python -m paper_2508_04257_b200.build --debug)")
    env = dict(os.environ, KVSINK_LIB=kv_build.DEBUG_LIB)
    r = subprocess.run([sys.executable, "-c", PROMPTS, ROOT], capture_output=True, text=True, env=env, timeout=600)
    assert r.returncode == 0 and "debug prompts ok" in r.stdout, r.stdout[-1500:] + r.stderr[-3000:]


FAILING_APPEND = r"""
import sys
sys.path.insert(0, sys.argv[1]); sys.path.insert(0, sys.argv[1] + "/tests")
import torch
import oracle
import paper_2508_04257_b200 as kv
from paper_2508_04257_b200 import binding, synth
from parity_util import compare_cache, configs, np16
TINY = synth.WORKLOADS["tiny"]
# bulk, streaming and generic kernels for the whole groups; the chunk ends the open group and leaves a remainder behind its last group
for bits, d, group in ((3, 128, 64), (2, 128, 128), (2, 128, 32), (4, 64, 80)):
    wl = TINY.scaled(bits=bits, head_dim=d, group=group, n_q_heads=4, n_kv_heads=2, batch=2, seq=4 * group, topk=9, pfn_n=1, seed=51 + bits)
    ocfg, gcfg = configs(wl)
    H, (K, V) = synth.make_hidden(wl, "cuda"), synth.make_kv(wl, 0, "cuda")
    gc = kv.KVCache(gcfg, kv.predict_sinks(gcfg, H, kv.SinkSet(gcfg)))
    oc = oracle.Cache(ocfg, *oracle.predict_sinks(ocfg, np16(H)))
    cut, end = group // 2 + 3, 3 * group + group // 2
    k, v = K[:, :, cut:end], V[:, :, cut:end]
    kv.quantize_append(gcfg, gc, K[:, :, :cut], V[:, :, :cut])
    before = binding.lib().kvsink_launch_count()
    binding.lib().kvsink_debug_fail_host_call(1)
    try:
        kv.quantize_append(gcfg, gc, k, v)
        raise SystemExit("the append did not report the failed call")
    except kv.KvsinkError as e:
        assert e.code == -7, e
    assert gc.seq_len == cut and binding.lib().kvsink_launch_count() == before
    kv.quantize_append(gcfg, gc, k, v)             # once more, and this time it works
    oracle.quantize_append(ocfg, oc, np16(K[:, :, :cut]), np16(V[:, :, :cut]))
    oracle.quantize_append(ocfg, oc, np16(k), np16(v))
    compare_cache(gc, oc, wl)
    assert kv.read_status(gc) == 0
print("failed append ok")
"""


@pytest.mark.gpu
def test_an_append_that_fails_on_the_host_leaves_the_open_group():
    if not os.path.exists(kv_build.DEBUG_LIB):
        pytest.skip("libkvsink_debug.so has not been built (python -m paper_2508_04257_b200.build --debug)")
    env = dict(os.environ, KVSINK_LIB=kv_build.DEBUG_LIB)
    r = subprocess.run([sys.executable, "-c", FAILING_APPEND, ROOT], capture_output=True, text=True, env=env, timeout=600)
    assert r.returncode == 0 and "failed append ok" in r.stdout, r.stdout[-1500:] + r.stderr[-3000:]
