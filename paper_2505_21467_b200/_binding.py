"""Binding of libdlm.so: argument marshalling only.

Every function has the name and the argument order of its C counterpart in include/dlm.h.
Tensors are torch CUDA tensors (PyTorch is used for device memory and streams only); each
call passes raw device pointers and the current CUDA stream.  The calls that enqueue kernels come
from the native module _dlm_calls (csrc/py_calls.cpp); context, size and diagnostic calls go through
ctypes.  There is no fallback: if the library is missing or a call fails, an exception is raised.
"""
from __future__ import annotations

import ctypes
import os

import torch

from . import build as _build

DLM_OK = 0
DLM_ERR_NULL, DLM_ERR_SHAPE, DLM_ERR_UNSUPPORTED, DLM_ERR_CAPACITY = -1, -2, -3, -4
DLM_ERR_WORKSPACE, DLM_ERR_CUDA, DLM_ERR_TIMEOUT, DLM_ERR_INDEX, DLM_ERR_DEVICE = -5, -6, -7, -8, -9
DLM_DST_APPEND, DLM_DST_WINDOW = 0, 1


class DlmError(RuntimeError):
    def __init__(self, code, where):
        self.code = code
        super().__init__(f"{where}: {dlm_strerror(code)} ({code})")


class dlm_kv_cache(ctypes.Structure):
    _fields_ = [("k", ctypes.c_void_p), ("v", ctypes.c_void_p), ("cache_len", ctypes.c_void_p),
                ("n_layers", ctypes.c_int32), ("batch", ctypes.c_int32), ("n_kv_heads", ctypes.c_int32),
                ("capacity", ctypes.c_int32), ("head_dim", ctypes.c_int32)]


_lib = None


def lib() -> ctypes.CDLL:
    """Loads libdlm.so (in-tree).  Raises if it has not been built."""
    global _lib
    if _lib is not None:
        return _lib
    path = _build.LIB
    if not os.path.exists(path):
        raise ImportError(f"{path} is missing: run `python -m paper_2505_21467_b200.build` "
                          "(there is no CPU or PyTorch fallback)")
    L = ctypes.CDLL(path)
    vp, i32, sz, u64, ip = ctypes.c_void_p, ctypes.c_int, ctypes.c_size_t, ctypes.c_uint64, ctypes.POINTER(ctypes.c_int)
    cache = ctypes.POINTER(dlm_kv_cache)
    for name, restype, argtypes in (
            ("dlm_create", i32, [ctypes.POINTER(vp), i32]),
            ("dlm_destroy", i32, [vp]),
            ("dlm_get_status", i32, [vp, vp]),
            ("dlm_strerror", ctypes.c_char_p, [i32]),
            ("dlm_launch_count", ctypes.c_int64, [vp]),
            ("dlm_attn_workspace_bytes", sz, [vp, cache, i32, i32, i32]),
            ("dlm_unmask_workspace_bytes", sz, [vp, i32, i32, i32]),
            ("dlm_unmask_scored_workspace_bytes", sz, [vp, i32, i32, i32]),
            ("dlm_window_proj_workspace_bytes", sz, [vp, i32, i32, i32]),
            ("dlm_selftest_wait_timeout", i32, [vp, u64, vp]),
            ("dlm_selftest_set_wait_limit", i32, [vp, u64]),
            ("dlm_selftest_set_attn_team_max", i32, [vp, i32, i32]),
            ("dlm_selftest_attn_schedule", i32, [vp, cache, i32, i32, i32, i32, ip, ip, ip, ip])):
        f = getattr(L, name)
        f.restype, f.argtypes = restype, argtypes
    _lib = L
    return L


def dlm_strerror(code: int) -> str:
    return lib().dlm_strerror(int(code)).decode()


def _check(code, where):
    if code != DLM_OK:
        raise DlmError(code, where)


def _ptr(t, dtype=None):
    if t is None:
        return None
    if not (isinstance(t, torch.Tensor) and t.is_cuda and t.is_contiguous()):
        raise TypeError("expected a contiguous CUDA tensor")
    if dtype is not None and t.dtype != dtype:
        raise TypeError(f"expected dtype {dtype}, got {t.dtype}")
    return ctypes.c_void_p(t.data_ptr())


def _stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


def dlm_create(device: int = 0) -> ctypes.c_void_p:
    ctx = ctypes.c_void_p()
    _check(lib().dlm_create(ctypes.byref(ctx), int(device)), "dlm_create")
    return ctx


def dlm_destroy(ctx) -> None:
    _check(lib().dlm_destroy(ctx), "dlm_destroy")


def dlm_get_status(ctx) -> int:
    """Synchronises the current stream; returns (and clears) the first device-side error code."""
    return int(lib().dlm_get_status(ctx, _stream()))


def dlm_launch_count(ctx) -> int:
    return int(lib().dlm_launch_count(ctx))


def make_kv_cache(k: torch.Tensor, v: torch.Tensor, cache_len: torch.Tensor) -> dlm_kv_cache:
    """View of caller-owned tensors: k, v bf16 [NL,B,Hkv,Lcap,D]; cache_len int32 [B]."""
    if k.dtype != torch.bfloat16 or k.shape != v.shape or k.dim() != 5:
        raise TypeError("k and v must be bf16 tensors of the same 5-d shape")
    NL, B, Hkv, Lcap, D = k.shape
    if cache_len.shape != (B,):
        raise TypeError("cache_len must have shape [batch]")
    c = dlm_kv_cache(_ptr(k).value, _ptr(v).value, _ptr(cache_len, torch.int32).value, NL, B, Hkv, Lcap, D)
    c._keepalive = (k, v, cache_len)
    return c


def dlm_attn_workspace_bytes(ctx, cache, n_layers_in_call, n_q_heads, q_cap) -> int:
    return int(lib().dlm_attn_workspace_bytes(ctx, ctypes.byref(cache), int(n_layers_in_call), int(n_q_heads),
                                              int(q_cap)))


def dlm_selftest_attn_schedule(ctx, cache, n_layers_in_call, n_q_heads, q_cap, cache_len_hint=0) -> dict:
    g, c, w, r = ctypes.c_int(), ctypes.c_int(), ctypes.c_int(), ctypes.c_int()
    _check(lib().dlm_selftest_attn_schedule(ctx, ctypes.byref(cache), int(n_layers_in_call), int(n_q_heads), int(q_cap),
                                            int(cache_len_hint), ctypes.byref(g), ctypes.byref(c), ctypes.byref(w),
                                            ctypes.byref(r)), "dlm_selftest_attn_schedule")
    return {"grid": g.value, "team": c.value, "whole_units": w.value, "chunk_rows": r.value}


def dlm_unmask_workspace_bytes(ctx, batch, block_len, vocab) -> int:
    return int(lib().dlm_unmask_workspace_bytes(ctx, int(batch), int(block_len), int(vocab)))


DLM_SCORE_CONFIDENCE, DLM_SCORE_NEG_ENTROPY, DLM_SCORE_MARGIN, DLM_SCORE_LOG_CONF_PLUS_NOISE = 0, 1, 2, 3


def dlm_unmask_scored_workspace_bytes(ctx, batch, block_len, vocab) -> int:
    return int(lib().dlm_unmask_scored_workspace_bytes(ctx, int(batch), int(block_len), int(vocab)))


def dlm_window_proj_workspace_bytes(ctx, rows, n_out, k_total) -> int:
    return int(lib().dlm_window_proj_workspace_bytes(ctx, int(rows), int(n_out), int(k_total)))


def dlm_selftest_set_wait_limit(ctx, limit_ns: int) -> None:
    _check(lib().dlm_selftest_set_wait_limit(ctx, ctypes.c_uint64(int(limit_ns))), "dlm_selftest_set_wait_limit")


def dlm_selftest_set_attn_team_max(ctx, max_blocks: int, force: bool = False) -> None:
    _check(lib().dlm_selftest_set_attn_team_max(ctx, int(max_blocks), int(force)), "dlm_selftest_set_attn_team_max")


def dlm_selftest_wait_timeout(ctx, limit_ns: int) -> None:
    _check(lib().dlm_selftest_wait_timeout(ctx, ctypes.c_uint64(int(limit_ns)), _stream()), "dlm_selftest_wait_timeout")


# The enqueueing calls.  They are bound to the native functions themselves once _dlm_calls can be loaded; until then (the
# package is imported by its own build) to stand-ins that load it at the first call or raise.
_calls = None


def _load_calls():
    global _calls
    if _calls is None:
        lib()   # the missing-library message, and the one copy of libdlm.so
        if os.path.exists(_build.CALLS) and not _build.calls_loadable():
            raise ImportError(f"{_build.CALLS} was not built from its present sources for {_build.calls_abi()}, whose objects it "
                              "would read: run `python -m paper_2505_21467_b200.build`")
        try:
            from . import _dlm_calls as m
        except ImportError as e:
            raise ImportError(f"{_build.CALLS} cannot be loaded ({e}): run `python -m paper_2505_21467_b200.build` "
                              "(there is no CPU or PyTorch fallback)") from e
        m.set_error(DlmError)
        m.set_types(ctypes.c_void_p, dlm_kv_cache)
        _calls = m
    return _calls


def _stand_in(name):
    def call(*args, **kwargs):
        return getattr(_load_calls(), name)(*args, **kwargs)
    call.__name__ = call.__qualname__ = name
    return call


try:
    _load_calls()
except ImportError:
    pass
for _name in ("dlm_kv_cache_commit", "dlm_freecache_attn_step", "dlm_unmask_select", "dlm_unmask_select_static",
              "dlm_unmask_select_scored", "dlm_guided_accept", "dlm_guided_accept_topk", "dlm_guided_accept_threshold",
              "dlm_window_qkv_project", "dlm_window_qkv_project_rope", "dlm_window_qkv_project_stage", "dlm_window_out_project"):
    globals()[_name] = getattr(_calls, _name) if _calls is not None else _stand_in(_name)
