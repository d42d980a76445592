"""Host-side checks of the C ABI that need no GPU: the library loads, exports every symbol
the header declares, sizes workspaces and rejects bad arguments before touching CUDA."""
import ctypes as C
import os
import re

import pytest

from paper_2510_20707_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.load_library()


def test_every_declared_symbol_is_exported(lib):
    header = open(os.path.join(ROOT, "include", "mixkv.h")).read()
    declared = set(re.findall(r"\b(mixkv_[a-z_]+)\s*\(", header))
    assert declared == set(binding.EXPORTS)
    for name in declared:
        assert getattr(lib, name) is not None


def test_status_strings(lib):
    assert binding.status_string(0) == "ok"
    assert "workspace" in binding.status_string(-3)
    assert "unknown" in binding.status_string(-99)


def test_default_params(lib):
    p = binding._CParams()
    lib.mixkv_default_params(C.byref(p), 4, 7, 128)
    assert (p.kv_heads, p.gqa_ratio, p.head_dim, p.window, p.pool_kernel, p.budget) == (4, 7, 128, 32, 7, 128)
    assert p.use_vnorm == 1 and p.mix_mode == 0 and abs(p.eps - 1e-6) < 1e-12


def test_workspace_size_grows_with_tokens():
    p = binding.Params(kv_heads=4, gqa_ratio=7, budget=128)
    a = binding.workspace_size(p, 1, 4096, 4096)
    b = binding.workspace_size(p, 1, 32768, 32768)
    c = binding.workspace_size(p, 8, 40960, 8192)
    assert 0 < a < b < c < 64 << 20


@pytest.mark.parametrize("kw,status", [
    (dict(pool_kernel=4), -1), (dict(budget=32), -1), (dict(budget=8), -1),
    (dict(head_dim=64), -2), (dict(gqa_ratio=8), -2), (dict(window=24, gqa_ratio=1), -2),
    (dict(mix_mode=7), -1), (dict(ada_floor=1.5), -1), (dict(kv_heads=0), -1),
])
def test_bad_params_are_rejected(kw, status):
    base = dict(kv_heads=4, gqa_ratio=7, budget=64)
    base.update(kw)
    with pytest.raises(binding.MixKVError) as e:
        binding.workspace_size(binding.Params(**base), 1, 1024, 1024)
    assert e.value.status == status


def test_entry_points_validate_before_any_cuda_call(lib):
    # null tensors, short sequences, bad offsets, small workspace: all host-side errors
    p = binding.Params(kv_heads=4, gqa_ratio=7, budget=64).c()
    ws = C.create_string_buffer(1 << 20)
    wsp = C.cast(ws, C.c_void_p).value
    wsp = (wsp + 255) // 256 * 256
    one = C.c_void_p(256)  # a non-null, aligned fake pointer; never dereferenced on error paths
    args = lambda L, wbytes, cu=None, batch=1: (one, one, one, cu, batch, L, C.byref(p), wsp, wbytes,
                                                None, one, one, one, None, None, None, None, None, None)
    assert lib.mixkv_compress_layer(*args(32, 1 << 19)) == -1           # L <= W
    assert lib.mixkv_compress_layer(*args(1024, 1024)) == -3            # workspace too small
    cu = (C.c_int32 * 3)(0, 500, 400)
    assert lib.mixkv_compress_layer(*args(0, 1 << 19, cu, 2)) == -1     # offsets not ascending
    assert lib.mixkv_compress_layer(*args(1024, 1 << 19, None, 2)) == -1  # batch > 1 needs offsets
    assert lib.mixkv_scores(None, one, one, None, 1, 1024, C.byref(p), wsp, 1 << 19, one, None,
                            None, None, None, None, None) == -1
    assert lib.mixkv_select(None, None, 1, 1024, C.byref(p), wsp, 1 << 19, one, one, one, None,
                            None) == -1


def test_stage_names_follow_the_route(lib):
    p = binding.Params(kv_heads=4, gqa_ratio=7, budget=256)
    assert binding.stage_names_for(p, 28, 1, 32768) == ["pass1", "pass2", "tail"]
    # one head-layer of 140000 candidates does not fit the tail kernel's shared memory
    assert binding.stage_names_for(p, 1, 1, 140032) == ["pass1", "pass2", "mixpool", "tail"]
    # 112 units of 65504 candidates: too long for one CTA per head, clusters of eight keep them
    assert binding.stage_names_for(p, 28, 1, 65536) == ["pass1", "pass2", "tail"]
    pa = binding.Params(kv_heads=4, gqa_ratio=7, budget=128, budget_mode=1)
    assert binding.stage_names_for(pa, 28, 8, 8192) == ["pass1", "pass2", "mixpool", "budget", "tail"]
    assert binding.stage_names(p) == ["pass1", "pass2", "tail"]


def test_device_check_without_a_device_or_with_one(lib):
    # no GPU here: the query fails and the entry point says so; on a B200 it reports 10.x
    import torch
    rc, major = binding.device_check()
    if torch.cuda.is_available():
        assert (rc, major) == (0, 10)
    else:
        assert rc == -4 and major == 0


@pytest.mark.parametrize("cu", [[], [0], [0, 64, 40], [0, 8]])
def test_binding_refuses_offsets_without_a_sequence(lib, cu):
    # no sequence, one offset, a descending one, one shorter than the window: refused before anything is allocated
    import torch
    K = torch.zeros((2, 64, 128), dtype=torch.bfloat16)
    p = binding.Params(kv_heads=2, gqa_ratio=1, window=16, budget=32)
    with pytest.raises(binding.MixKVError) as e:
        out = {k: torch.zeros(4) for k in ("K_out", "V_out", "out_row_offsets", "status")}
        ws = None if len(cu) < 2 else torch.zeros(1 << 20, dtype=torch.uint8)
        binding.compress_layer(K, K, torch.zeros((1, 2, 16, 128), dtype=torch.bfloat16), p, cu_seqlens=cu, out=out,
                               workspace=ws, stream=type("S", (), {"cuda_stream": 0}))
    assert e.value.status == -1


def test_binding_passes_on_what_a_truth_value_raises(lib):
    import numpy as np
    import torch
    K = torch.zeros((2, 64, 128), dtype=torch.bfloat16)
    p = binding.Params(kv_heads=2, gqa_ratio=1, window=16, budget=32)
    with pytest.raises(ValueError):     # the truth value of an array is ambiguous
        binding.scores(K, K, torch.zeros((1, 2, 16, 128), dtype=torch.bfloat16), p, want_parts=np.ones(2))


@pytest.mark.parametrize("block", [0, -3, 1 << 31, (1 << 32) + 16])
def test_binding_refuses_block_sizes_the_library_cannot_take(lib, block):
    import torch
    with pytest.raises(binding.MixKVError) as e:
        binding.similarity_map(torch.zeros((1, 64, 128), dtype=torch.bfloat16), block)
    assert e.value.status == -1


@pytest.mark.parametrize("kw", [dict(kv_heads=(1 << 32) + 2), dict(gqa_ratio=1 - (1 << 32)), dict(max_rows=(1 << 32) + 100),
                                dict(max_rows=1 << 31)])
def test_binding_refuses_decode_sizes_the_library_cannot_take(lib, kw):
    # (the lower 32 bits of each are sizes that it would take)
    import torch
    cache, offs = torch.zeros((1, 8, 128), dtype=torch.bfloat16), torch.zeros((1, 3), dtype=torch.int32)
    with pytest.raises(binding.MixKVError) as e:
        binding.decode_attention(cache, cache, offs, cache[:, None, :2], **dict(dict(kv_heads=2, gqa_ratio=1, max_rows=4), **kw))
    assert e.value.status == -1


@pytest.mark.parametrize("kw,cu", [(dict(kv_heads=(1 << 32) + 2), None), (dict(budget=(1 << 32) + 32), None),
                                   (dict(pool_kernel=7 - (1 << 32)), None), ({}, [0, (1 << 32) + 64])])
def test_binding_refuses_params_and_offsets_the_library_cannot_take(lib, kw, cu):
    import torch
    K, Q = torch.zeros((2, 64, 128), dtype=torch.bfloat16), torch.zeros((1, 2, 16, 128), dtype=torch.bfloat16)
    p = binding.Params(**dict(dict(kv_heads=2, gqa_ratio=1, window=16, budget=32), **kw))
    for call in (lambda: binding.scores(K, K, Q, p, cu_seqlens=cu), lambda: binding.compress_layer(K, K, Q, p, cu_seqlens=cu),
                 lambda: binding.compress_layers(K[None], K[None], Q[None], p, cu_seqlens=cu),
                 lambda: binding.select(torch.zeros((2, 48)), p, cu_seqlens=cu)):
        with pytest.raises(binding.MixKVError) as e:
            call()
        assert e.value.status == -1


def test_native_binding_is_rebuilt_for_another_torch(lib, monkeypatch):
    # the module is compiled against torch's C++ interface: a file newer than its sources does not show that
    assert build.host_matches() and not build.host_is_stale()
    tag = build.host_tag()
    monkeypatch.setattr(build, "host_tag", lambda: tag.replace("torch-", "torch-x"))
    assert build.host_is_stale()
    monkeypatch.setattr(binding, "_host_module", None)
    with pytest.raises(ImportError):
        binding._host()
