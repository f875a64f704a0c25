"""Host-side checks of the C ABI: the library loads, exports every declared symbol, and rejects
bad arguments before touching the GPU."""
import ctypes
import os
import re

import pytest

from paper_2506_11498_b200 import build as lib_build
from paper_2506_11498_b200 import lrsa

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_build.build()


def declared_symbols():
    text = open(os.path.join(ROOT, "include", "lrsa.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(lrsa_[a-z_0-9]+)\s*\(", text)))


def test_exports_every_declared_symbol():
    names = declared_symbols()
    assert {"lrsa_score_select", "lrsa_attn_fwd", "lrsa_attn_bwd", "lrsa_workspace_bytes"} <= set(names)
    L = ctypes.CDLL(lrsa.LIB_PATH)
    for n in names:
        assert hasattr(L, n), n


def test_status_strings():
    assert lrsa.status_string(0) == "ok"
    assert "workspace" in lrsa.status_string(3)
    assert lrsa.status_string(99) == "unknown status"


GOOD = dict(batch=1, n_q_heads=4, n_kv_heads=2, seq_len=1000, head_dim=128, lag=128, top_k=32, n_sink=4)


@pytest.mark.parametrize("change,status", [
    ({}, 0),
    ({"batch": 0}, 1), ({"n_q_heads": 3}, 1), ({"top_k": 129}, 1), ({"top_k": 0}, 1), ({"n_sink": -1}, 1),
    ({"std_ddof": 2}, 1), ({"n_dense_prev": 2}, 1), ({"softmax_scale": -1.0}, 1),
    ({"head_dim": 96}, 2), ({"chunk": 64}, 2), ({"seq_len": 3}, 2), ({"lag": 40000, "top_k": 5, "seq_len": 100000}, 2),
])
def test_parameter_validation(change, status):
    p = lrsa.Params(**{**GOOD, **change})
    if status == 0:
        a, b, c = lrsa.lrsa_workspace_bytes(p)
        assert a >= 256 and b >= 256 and c >= 256
        assert lrsa.lrsa_num_sel_windows(p) == (1000 - 4) // 128 - 1
    else:
        with pytest.raises(lrsa.LrsaError) as e:
            lrsa.lrsa_workspace_bytes(p)
        assert e.value.status == status


def test_null_and_misaligned_pointers_are_rejected_on_the_host():
    L = lrsa.lib()
    cp = lrsa.Params(**GOOD).c()
    null = ctypes.c_void_p(0)
    fake = ctypes.c_void_p(0x10000)      # never dereferenced: validation fails first
    odd = ctypes.c_void_p(0x10008)
    assert L.lrsa_score_select(ctypes.byref(cp), null, fake, fake, null, fake, 1 << 30, null) == 1
    assert L.lrsa_score_select(ctypes.byref(cp), odd, fake, fake, null, fake, 1 << 30, null) == 1
    assert L.lrsa_score_select(ctypes.byref(cp), fake, fake, fake, null, fake, 16, null) == 3
    assert L.lrsa_attn_fwd(ctypes.byref(cp), fake, fake, fake, fake, null, fake, fake, 1 << 30, null) == 1
    assert L.lrsa_attn_fwd(ctypes.byref(cp), fake, fake, fake, fake, fake, fake, fake, 0, null) == 3
    assert L.lrsa_attn_bwd(ctypes.byref(cp), fake, fake, fake, fake, fake, fake, fake, fake, fake, null, fake,
                           1 << 30, null) == 1
    assert L.lrsa_attn_bwd(ctypes.byref(cp), fake, fake, fake, fake, fake, fake, fake, fake, fake, fake, fake,
                           0, null) == 3
    assert L.lrsa_workspace_status(null, null) == 1


def test_geometry_matches_definition():
    for N, S, L, want in ((32768, 4, 1024, 30), (4096, 16, 512, 6), (9, 1, 2, 3), (300, 4, 256, 0), (516, 4, 256, 1)):
        p = lrsa.Params(1, 1, 1, N, 64, L, 1, S)
        assert lrsa.lrsa_num_sel_windows(p) == want


def test_packed_parameter_validation():
    ok = lrsa.Params(**GOOD, cu_seqlens=(0, 300, 1000))
    assert lrsa.lrsa_num_sel_windows(ok) == ((300 - 4) // 128 - 1) + ((700 - 4) // 128 - 1)
    for bad in ((1, 300, 1000), (0, 300, 900), (0, 300, 300, 1000), (0, 1200, 1000)):
        with pytest.raises(lrsa.LrsaError) as e:
            lrsa.lrsa_num_sel_windows(lrsa.Params(**GOOD, cu_seqlens=bad))
        assert e.value.status == 1
    assert lrsa.lrsa_num_sel_windows(lrsa.Params(**{**GOOD, "chunk": 256})) == (1000 - 4) // 128 - 1


def test_o_residual_must_be_16_byte_aligned():
    import ctypes
    out = ctypes.c_int32(0)
    cp = lrsa.Params(**GOOD).c()
    cp.o_residual = 4096
    assert lrsa.lib().lrsa_num_sel_windows(ctypes.byref(cp), ctypes.byref(out)) == 0
    cp.o_residual = 4096 + 8
    assert lrsa.lib().lrsa_num_sel_windows(ctypes.byref(cp), ctypes.byref(out)) == 1


@pytest.mark.parametrize("shape", [dict(), dict(seq_len=32768, n_q_heads=28, n_kv_heads=4, lag=1024, top_k=256),
                                   dict(seq_len=32768, head_dim=64, lag=256, top_k=64, n_sink=16), dict(seq_len=700, lag=500, n_sink=40)])
def test_workspace_sizes_do_not_depend_on_the_packing(shape):
    """A workspace sized for one batch of a data loader serves the next: the sizes follow the row's shape alone."""
    import random
    args = {**GOOD, **shape}
    want = lrsa.lrsa_workspace_bytes(lrsa.Params(**args))
    n, r = args["seq_len"], random.Random(5)
    for cuts in ([], [n // 2], range(16, n, 16), range(1, 18), sorted(r.sample(range(1, n), 15)), sorted(r.sample(range(1, n), 40))):
        assert lrsa.lrsa_workspace_bytes(lrsa.Params(**args, cu_seqlens=(0, *cuts, n))) == want


def test_dependent_launches_read_through_plain_loads():
    """A kernel that may start while the one in front of it still writes must not read that data through the read-only path
    (__ldg, ld.global.nc, which const __restrict__ pointers invite too): such loads are not ordered by griddepcontrol.wait."""
    csrc = os.path.join(ROOT, "paper_2506_11498_b200", "csrc")
    files = [f for f in os.listdir(csrc) if f.endswith(".cu") and "griddepcontrol.wait" in open(os.path.join(csrc, f)).read()]
    assert len(files) >= 6
    for f in files + ["attn_common_sm100.h", "attn_bwd_sm100.h", "sm100_ptx.h"]:
        code = re.sub(r"//[^\n]*", "", open(os.path.join(csrc, f)).read())
        for word in ("__ldg", "ld.global.nc", "__restrict__"):
            assert word not in code, (f, word)


def test_params_keep_their_value_semantics_after_a_call():
    """The struct that calls reuse is no part of the parameters: fields, equality, copies and pickles stay those of the fields."""
    import copy, dataclasses, pickle
    p = lrsa.Params(**GOOD, cu_seqlens=(0, 300, 1000))
    fields = dict(vars(p))
    n = lrsa.lrsa_num_sel_windows(p)
    assert vars(p) == fields and lrsa.Params(**vars(p)) == p
    for q in (copy.copy(p), copy.deepcopy(p), pickle.loads(pickle.dumps(p)), dataclasses.replace(p)):
        assert q == p and hash(q) == hash(p) and lrsa.lrsa_num_sel_windows(q) == n
    assert lrsa.lrsa_num_sel_windows(dataclasses.replace(p, n_sink=44)) == (300 - 44) // 128 - 1 + (700 - 44) // 128 - 1


def test_boundaries_in_a_list_are_read_at_each_call():
    p = lrsa.Params(**GOOD, cu_seqlens=[0, 300, 1000])
    for cut in (300, 500, 262):
        p.cu_seqlens[1] = cut
        assert lrsa.lrsa_num_sel_windows(p) == lrsa.lrsa_num_sel_windows(lrsa.Params(**GOOD, cu_seqlens=(0, cut, 1000)))


def test_threads_that_build_the_struct_together_hold_live_ones(monkeypatch):
    """Two threads find no struct yet and both build one: every address handed to the library is that of a live struct,
    in these calls and in later ones (the structs made in between take the place of one that was let go)."""
    import sys
    import threading
    import torch
    lrsa.lib()
    build, seen = lrsa.Params.c, []

    class Calls:                   # stands for the helper module: what the struct holds when the library reads it
        @staticmethod
        def cache_append(address, *rest):
            seen.append(lrsa.lrsa_params_t.from_address(address).seq_len)
            return 0

    t = torch.zeros(1, 2, 1, 128)
    stream = type("S", (), {"cuda_stream": 0})
    monkeypatch.setattr(lrsa, "_call", Calls)
    interval = sys.getswitchinterval()
    sys.setswitchinterval(1e-6)
    try:
        for _ in range(200):
            together = threading.Barrier(2)

            def slow(self, *a):
                cp = build(self, *a)
                together.wait(10)
                return cp

            monkeypatch.setattr(lrsa.Params, "c", slow)
            cache = lrsa.KVCache.__new__(lrsa.KVCache)
            cache.params, cache.buf, cache.ws, cache.n_tokens = lrsa.Params(**GOOD), t, t, 0
            threads = [threading.Thread(target=cache.append, args=(t, t, stream)) for _ in range(2)]
            [x.start() for x in threads]
            [x.join() for x in threads]
            others = [lrsa.lrsa_params_t() for _ in range(64)]
            cache.append(t, t, stream)
            del others
    finally:
        sys.setswitchinterval(interval)
    assert seen == [1000] * 600


def test_a_cache_works_in_a_process_that_has_made_no_call(monkeypatch):
    """As after unpickling: the library is loaded by the first append or decode.  A cache saved before a field was added
    works too.  (Calls that the library refuses before it touches the GPU.)"""
    import torch
    cache = lrsa.KVCache(lrsa.Params(**GOOD), device="cpu")
    for name in set(vars(cache)) - {"params", "buf", "ws", "n_tokens"}:
        delattr(cache, name)
    stream = type("S", (), {"cuda_stream": 0})
    k = torch.zeros((1, 2, 1, 128), dtype=torch.bfloat16)
    q = torch.zeros((1, 4, 128), dtype=torch.bfloat16)
    cache.n_tokens = 1000                     # full: one more token is an invalid argument
    for call in (lambda: cache.append(k, k, stream), lambda: cache.decode(q, stream=stream)):
        monkeypatch.setattr(lrsa, "_call", None)
        monkeypatch.setattr(lrsa, "_lib", None)
        with pytest.raises(lrsa.LrsaError) as e:
            call()
        assert e.value.status == 1
        cache.n_tokens = 0                    # nothing to decode


@pytest.mark.parametrize("name,content", [("_lrsa_call.so", None), ("_lrsa_call.so", "no module"), ("none", None)])
def test_the_library_works_without_its_helper_module(monkeypatch, tmp_path, name, content):
    """The module is built for one interpreter and only saves time: without it, or with one that does not load, every call is there."""
    import torch
    path = tmp_path / name
    if content:
        path.write_text(content)
    monkeypatch.setattr(lrsa, "CALL_PATH", str(path))
    monkeypatch.setattr(lrsa, "_lib", None)
    monkeypatch.setattr(lrsa, "_call", None)
    p = lrsa.Params(**GOOD)
    assert lrsa.lrsa_num_sel_windows(p) == (1000 - 4) // 128 - 1
    cache = lrsa.KVCache(p, device="cpu")
    cache.n_tokens = 1000
    k, q = torch.zeros((1, 2, 1, 128), dtype=torch.bfloat16), torch.zeros((1, 4, 128), dtype=torch.bfloat16)
    stream = type("S", (), {"cuda_stream": 0})
    with pytest.raises(lrsa.LrsaError) as e:      # refused by the library: the arguments arrived in their places
        cache.append(k, k, stream)
    assert e.value.status == 1
    cache.n_tokens = 0
    with pytest.raises(lrsa.LrsaError) as e:
        cache.decode(q, stream=stream)
    assert e.value.status == 1


def test_the_helper_module_is_rebuilt_when_it_is_the_older_one(monkeypatch, tmp_path):
    """Whatever the age of the library; and a build that fails leaves no older module behind."""
    path = tmp_path / "_lrsa_call.so"
    path.write_bytes(b"old")
    os.utime(path, (1, 1))
    monkeypatch.setattr(lib_build, "CALL", str(path))
    assert lib_build.call_is_stale()
    monkeypatch.setenv("CC", "false")
    lib_build.build()
    assert not path.exists()
    monkeypatch.delenv("CC")
    lib_build.build()
    assert path.exists() and not lib_build.call_is_stale()
