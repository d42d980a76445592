"""Python binding of the MixKV C ABI (``include/mixkv.h``).

Argument marshalling only: every function hands device pointers of torch tensors to the
library and returns the tensors it filled.  No arithmetic of the method happens here, and
nothing falls back to PyTorch ops or the CPU: if ``libmixkv.so`` is missing,
:func:`load_library` raises, and so does the first call that enqueues work without
``_mixkv_host.so``.

The calls that enqueue work go through the native module ``_mixkv_host``
(``csrc/host/host_binding.cpp``), the rest through ctypes, each to the entry point of the same
name but for :func:`scores`, :func:`scores_static` and :func:`select`, which take the variants of
``csrc/internal_api.h`` (the call itself clears the status word it hands out), and
:func:`compress_layer`, which is ``mixkv_compress_layer_traced`` with no events.

The calls may be made by several threads at once (the interpreter lock is given up inside them); a
``workspace`` then belongs to one of them at a time, on one stream too.

A call runs on ``stream`` (a torch stream; default: the current one), and what it allocates, its outputs
among it, belongs to that stream as if it were the current one: the caller orders other streams that read
the outputs behind it, and tells the allocator of them (``Tensor.record_stream``) before it lets go of them.
Inputs, like those of any call on another stream than their own, are the caller's to keep until it is done.
"""
from __future__ import annotations

import ctypes as C
import importlib.machinery
import importlib.util
import os
from dataclasses import dataclass
from typing import Dict, Optional, Sequence

import torch

_PKG = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_PKG, "libmixkv.so")
HOST_PATH = os.path.join(_PKG, "_mixkv_host.so")

EXPORTS = ("mixkv_default_params", "mixkv_workspace_size", "mixkv_scores", "mixkv_select",
           "mixkv_compress_layer", "mixkv_compress_layer_traced", "mixkv_launches_per_layer",
           "mixkv_stage_name", "mixkv_status_string", "mixkv_scores_static",
           "mixkv_workspace_size_layers", "mixkv_compress_layers",
           "mixkv_compress_layers_budgeted", "mixkv_layer_budget_schedule",
           "mixkv_similarity_workspace_size", "mixkv_similarity_map", "mixkv_decode_attention",
           "mixkv_selftest_bounded_wait", "mixkv_launches_for", "mixkv_stage_name_for",
           "mixkv_device_check")


class MixKVError(RuntimeError):
    def __init__(self, status: int, what: str):
        super().__init__(f"{what}: {status_string(status)} ({status})")
        self.status = status


class _CParams(C.Structure):
    _fields_ = [("kv_heads", C.c_int32), ("gqa_ratio", C.c_int32), ("head_dim", C.c_int32),
                ("window", C.c_int32), ("pool_kernel", C.c_int32), ("pool_mode", C.c_int32),
                ("use_vnorm", C.c_int32), ("mix_mode", C.c_int32), ("budget_mode", C.c_int32),
                ("budget", C.c_int32), ("ada_floor", C.c_float), ("eps", C.c_float),
                ("softmax_scale", C.c_float)]


@dataclass
class Params:
    """Mirror of ``mixkv_params`` (see include/mixkv.h for the meaning of each field)."""
    kv_heads: int
    gqa_ratio: int
    head_dim: int = 128
    window: int = 32
    pool_kernel: int = 7
    pool_mode: int = 0
    use_vnorm: int = 1
    mix_mode: int = 0
    budget_mode: int = 0
    budget: int = 64
    ada_floor: float = 0.2
    eps: float = 1e-6
    softmax_scale: float = 0.0

    def c(self) -> _CParams:
        return _CParams(self.kv_heads, self.gqa_ratio, self.head_dim, self.window,
                        self.pool_kernel, self.pool_mode, self.use_vnorm, self.mix_mode,
                        self.budget_mode, self.budget, self.ada_floor, self.eps,
                        self.softmax_scale)


_lib: Optional[C.CDLL] = None
_host_module = None


def load_library() -> C.CDLL:
    """Loads libmixkv.so from the package directory; raises if it has not been built."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise FileNotFoundError(
                f"{LIB_PATH} not found: build it with `python -m paper_2510_20707_b200.build` "
                "(there is no CPU or PyTorch fallback)")
        lib = C.CDLL(LIB_PATH)
        vp, i32, sz = C.c_void_p, C.c_int32, C.c_size_t
        lib.mixkv_status_string.restype = C.c_char_p
        lib.mixkv_status_string.argtypes = [C.c_int]
        lib.mixkv_default_params.restype = None
        lib.mixkv_default_params.argtypes = [C.POINTER(_CParams), i32, i32, i32]
        lib.mixkv_workspace_size.argtypes = [C.POINTER(_CParams), i32, C.c_int64, i32,
                                             C.POINTER(sz)]
        lib.mixkv_workspace_size_layers.argtypes = [C.POINTER(_CParams), i32, i32, C.c_int64, i32,
                                                    C.POINTER(sz)]
        lib.mixkv_launches_per_layer.argtypes = [C.POINTER(_CParams)]
        lib.mixkv_launches_for.argtypes = [C.POINTER(_CParams), i32, i32, i32]
        lib.mixkv_stage_name_for.argtypes = [C.POINTER(_CParams), i32, i32, i32, i32]
        lib.mixkv_stage_name_for.restype = C.c_char_p
        lib.mixkv_device_check.argtypes = [C.POINTER(i32)]
        lib.mixkv_scores.argtypes = [vp, vp, vp, C.POINTER(i32), i32, i32, C.POINTER(_CParams),
                                     vp, sz, vp, vp, vp, vp, vp, vp, vp]
        lib.mixkv_scores_static.argtypes = [vp, vp, vp, C.POINTER(i32), i32, i32,
                                            C.POINTER(_CParams), vp, vp, vp, vp, vp, vp, vp]
        lib.mixkv_select.argtypes = [vp, C.POINTER(i32), i32, i32, C.POINTER(_CParams), vp, sz,
                                     vp, vp, vp, vp, vp]
        lib.mixkv_compress_layer.argtypes = [vp, vp, vp, C.POINTER(i32), i32, i32,
                                             C.POINTER(_CParams), vp, sz, vp, vp, vp, vp, vp, vp,
                                             vp, vp, vp, vp]
        lib.mixkv_compress_layer_traced.argtypes = lib.mixkv_compress_layer.argtypes + [
            C.POINTER(vp), i32]
        lib.mixkv_compress_layers.argtypes = [vp, vp, vp, i32, C.c_int64, C.c_int64,
                                              C.POINTER(i32), i32, i32, C.POINTER(_CParams), vp,
                                              sz, vp, vp, vp, vp, vp, vp, vp, vp, vp, vp,
                                              C.POINTER(vp), i32]
        lib.mixkv_compress_layers_budgeted.argtypes = [
            vp, vp, vp, i32, C.c_int64, C.c_int64, C.POINTER(i32), i32, i32, C.POINTER(_CParams),
            vp, sz, vp, vp, vp, vp, vp, vp, vp, vp, vp, vp, vp]
        lib.mixkv_layer_budget_schedule.argtypes = [i32, i32, i32, i32, C.POINTER(i32)]
        lib.mixkv_similarity_workspace_size.argtypes = [i32, i32, i32, C.POINTER(sz)]
        lib.mixkv_similarity_map.argtypes = [vp, i32, i32, i32, i32, vp, sz, vp, vp, vp]
        lib.mixkv_decode_attention.argtypes = [vp, vp, vp, C.c_int64, vp, i32, i32, i32, i32, i32,
                                               C.c_float, i32, vp, vp]
        lib.mixkv_selftest_bounded_wait.argtypes = [vp, vp, vp]
        lib.mixkv_stage_name.restype = C.c_char_p
        lib.mixkv_stage_name.argtypes = [C.POINTER(_CParams), i32]
        _lib = lib
    return _lib


def status_string(status: int) -> str:
    return load_library().mixkv_status_string(int(status)).decode()


def _host():
    """The native half of the binding (loads the library first)."""
    global _host_module
    if _host_module is None:
        load_library()
        if not os.path.exists(HOST_PATH):
            raise FileNotFoundError(
                f"{HOST_PATH} not found: build it with `python -m paper_2510_20707_b200.build`")
        from . import build
        if not build.host_matches(HOST_PATH):
            raise ImportError(f"{HOST_PATH} was built for another torch or Python: build it again with "
                              "`python -m paper_2510_20707_b200.build`")
        loader = importlib.machinery.ExtensionFileLoader("_mixkv_host", HOST_PATH)
        spec = importlib.util.spec_from_file_location("_mixkv_host", HOST_PATH, loader=loader)
        module = importlib.util.module_from_spec(spec)
        loader.exec_module(module)
        module.setup(LIB_PATH, MixKVError)
        _host_module = module
    return _host_module


def _stream(stream) -> int:
    if stream is None:
        stream = torch.cuda.current_stream()
    return stream.cuda_stream


def _events(trace_events):
    """Address and length of a ctypes array of cudaEvent_t handles (see mixkv_compress_layer_traced)."""
    return (0, 0) if trace_events is None else (C.addressof(trace_events), len(trace_events))


def workspace_size(params: Params, batch: int, total_tokens: int, max_seq_len: int) -> int:
    out = C.c_size_t(0)
    pc = params.c()
    rc = load_library().mixkv_workspace_size(C.byref(pc), batch, total_tokens, max_seq_len,
                                             C.byref(out))
    if rc != 0:
        raise MixKVError(rc, "mixkv_workspace_size")
    return int(out.value)


def workspace_size_layers(params: Params, n_layers: int, batch: int, total_tokens: int,
                          max_seq_len: int) -> int:
    out = C.c_size_t(0)
    pc = params.c()
    rc = load_library().mixkv_workspace_size_layers(C.byref(pc), n_layers, batch, total_tokens,
                                                    max_seq_len, C.byref(out))
    if rc != 0:
        raise MixKVError(rc, "mixkv_workspace_size_layers")
    return int(out.value)


def launches_per_layer(params: Params) -> int:
    pc = params.c()
    return int(load_library().mixkv_launches_per_layer(C.byref(pc)))


def stage_names(params: Params):
    pc = params.c()
    lib = load_library()
    return [lib.mixkv_stage_name(C.byref(pc), i).decode() for i in range(launches_per_layer(params))]


def stage_names_for(params: Params, n_layers: int, batch: int, max_seq_len: int):
    """Names of the kernels a call of this shape enqueues when it is given ``trace_events``
    (mixkv_launches_for / mixkv_stage_name_for): the route depends on the longest sequence and the
    number of units.  Without events, calls of few heads with adaptive budgets take another one (mix,
    budgets and selection in one kernel, the same results): their tail cannot be timed with events."""
    pc = params.c()
    lib = load_library()
    n = int(lib.mixkv_launches_for(C.byref(pc), n_layers, batch, max_seq_len))
    return [lib.mixkv_stage_name_for(C.byref(pc), n_layers, batch, max_seq_len, i).decode()
            for i in range(n)]


def device_check():
    """mixkv_device_check: (status, major compute capability of the current device)."""
    major = C.c_int32(0)
    rc = int(load_library().mixkv_device_check(C.byref(major)))
    return rc, int(major.value)


def scores(K: torch.Tensor, V: Optional[torch.Tensor], Q: torch.Tensor, params: Params,
           cu_seqlens: Optional[Sequence[int]] = None, rbar_in: Optional[torch.Tensor] = None,
           workspace: Optional[torch.Tensor] = None, stream=None,
           want_parts: bool = True) -> Dict[str, torch.Tensor]:
    """mixkv_scores: K, V [H, Ltot, 128] bf16, Q [batch, H*G, W, 128] bf16 (device tensors)."""
    return (_host_module or _host()).scores(K, V, Q, params, cu_seqlens, rbar_in, workspace, stream,
                                            want_parts, False)


def scores_static(K: torch.Tensor, V: Optional[torch.Tensor], Q: torch.Tensor, params: Params,
                  cu_seqlens: Optional[Sequence[int]] = None,
                  rbar_in: Optional[torch.Tensor] = None, stream=None) -> Dict[str, torch.Tensor]:
    """mixkv_scores_static: the same scores as :func:`scores`, for callers that cannot give
    the library a workspace.  The scratch the kernels need lives inside the library (a fixed
    array, see MIXKV_STATIC_SCRATCH_BYTES in the header), so this function hands over inputs
    and outputs only; the output tensors below are the caller's, as in :func:`scores`.
    Raises MixKVError (status -6) when the problem is too large for the built-in array.
    Calls on one device share that array: do not let two of them overlap on the GPU (several
    threads may call with one stream)."""
    return (_host_module or _host()).scores(K, V, Q, params, cu_seqlens, rbar_in, None, stream, True,
                                            True)


def select(s: torch.Tensor, params: Params, cu_seqlens: Optional[Sequence[int]] = None,
           workspace: Optional[torch.Tensor] = None, stream=None) -> Dict[str, torch.Tensor]:
    """mixkv_select on scores [H, Ptot] fp32 (device tensor)."""
    return (_host_module or _host()).select(s, params, cu_seqlens, workspace, stream)


def compress_layer(K: torch.Tensor, V: torch.Tensor, Q: torch.Tensor, params: Params,
                   cu_seqlens: Optional[Sequence[int]] = None,
                   rbar_in: Optional[torch.Tensor] = None,
                   workspace: Optional[torch.Tensor] = None, stream=None,
                   out: Optional[Dict[str, torch.Tensor]] = None,
                   want_aux: bool = True, trace_events=None) -> Dict[str, torch.Tensor]:
    """mixkv_compress_layer.  Returns K_out / V_out [batch*H*B, 128] (rows beyond
    out_row_offsets[-1] are untouched), out_row_offsets and, if want_aux, idx / counts /
    idx_offsets / s_comp.  `out` lets a caller reuse output tensors across calls.  `trace_events`: a
    ctypes array of cudaEvent_t handles, recorded around the kernels of :func:`stage_names_for`."""
    events, n_events = (0, 0) if trace_events is None else _events(trace_events)
    return (_host_module or _host()).compress_layer(K, V, Q, params, cu_seqlens, rbar_in, workspace, stream,
                                                    out, want_aux, events, n_events)


def compress_layers(K: torch.Tensor, V: torch.Tensor, Q: torch.Tensor, params: Params,
                    cu_seqlens: Optional[Sequence[int]] = None,
                    rbar_in: Optional[torch.Tensor] = None,
                    workspace: Optional[torch.Tensor] = None, stream=None,
                    out: Optional[Dict[str, torch.Tensor]] = None,
                    want_aux: bool = True, trace_events=None,
                    head_budgets: Optional[torch.Tensor] = None) -> Dict[str, torch.Tensor]:
    """mixkv_compress_layers: K, V [n_layers, H, Ltot, 128], Q [n_layers, batch, H*G, W, 128]
    (bf16 device tensors; the layer dimension may be strided, the rest contiguous).  Returns
    K_out / V_out [n_layers, batch*H*B, 128], out_row_offsets [n_layers, batch*H+1] and, if
    want_aux, idx [n_layers, cap] / counts / idx_offsets / s_comp.  With head_budgets (int32
    device tensor [n_layers, batch*H], rows to keep per head, window included) the call goes to
    mixkv_compress_layers_budgeted."""
    events, n_events = (0, 0) if trace_events is None else _events(trace_events)
    return (_host_module or _host()).compress_layers(K, V, Q, params, cu_seqlens, rbar_in, workspace, stream,
                                                     out, want_aux, events, n_events, head_budgets)


def layer_budget_schedule(n_layers: int, budget: int, window: int, taper_permille: int):
    """mixkv_layer_budget_schedule: rows to keep per head of each layer (host list), falling
    linearly with depth, total n_layers * budget."""
    arr = (C.c_int32 * n_layers)()
    rc = load_library().mixkv_layer_budget_schedule(n_layers, budget, window, taper_permille, arr)
    if rc != 0:
        raise MixKVError(rc, "mixkv_layer_budget_schedule")
    return [int(v) for v in arr]


def similarity_map(X: torch.Tensor, block: int, want_mean: bool = True, stream=None):
    """mixkv_similarity_map: X [heads, L, 128] bf16 device tensor -> (cells [heads, T, T] fp32,
    mean [heads] fp32 or None): block-mean cosine similarity of the rows of every head.  (A cell
    that a wait inside the kernel ran out on is NaN: there is no status word.)"""
    return (_host_module or _host()).similarity_map(X, block, want_mean, stream)


def decode_attention(K_cache: torch.Tensor, V_cache: torch.Tensor, out_row_offsets: torch.Tensor,
                     q: torch.Tensor, kv_heads: int, gqa_ratio: int, max_rows: int,
                     softmax_scale: float = 0.0, stream=None) -> torch.Tensor:
    """mixkv_decode_attention: K_cache / V_cache [n_layers, rows_cap, 128] bf16 (the compact
    cache), out_row_offsets [n_layers, batch*H+1] int32, q [n_layers, batch, H*G, 128] bf16 ->
    [n_layers, batch, H*G, 128] fp32."""
    return (_host_module or _host()).decode_attention(K_cache, V_cache, out_row_offsets, q, kv_heads,
                                                      gqa_ratio, max_rows, softmax_scale, stream)


def selftest_bounded_wait(stream=None):
    """mixkv_selftest_bounded_wait: returns (status, seconds waited) after the kernel has ended."""
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    waited = torch.zeros(1, dtype=torch.int64, device="cuda")
    rc = load_library().mixkv_selftest_bounded_wait(status.data_ptr(), waited.data_ptr(),
                                                    _stream(stream))
    if rc != 0:
        raise MixKVError(rc, "mixkv_selftest_bounded_wait")
    torch.cuda.synchronize()
    return int(status.item()), int(waited.item()) * 1e-9
