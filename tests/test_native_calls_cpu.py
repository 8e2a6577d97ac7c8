"""The native entry points check and order their arguments like the Python signatures they stand for (no GPU needed)."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2505_21467_b200 as dlm
from paper_2505_21467_b200 import build as _build


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()


def _args():
    t = torch.zeros(4, dtype=torch.int32)
    return dict(ctx=None, tok_dlm=t, tok_ar=t, batch=1, block_len=4, masked=t, tokens=t, fallback_source=0, accept=t, acc_idx=t, n_acc=t)


def test_wrong_argument_counts_and_names():
    a = _args()
    with pytest.raises(TypeError, match="11 arguments"):
        dlm.dlm_guided_accept(None, a["tok_dlm"])
    with pytest.raises(TypeError, match="unexpected or repeated"):
        dlm.dlm_guided_accept(*list(a.values())[:-1], acc_idx=a["acc_idx"])
    with pytest.raises(TypeError, match="unexpected or repeated"):
        dlm.dlm_guided_accept(*list(a.values())[:-1], nonsense=1)


def test_tensors_are_checked_before_anything_runs():
    a = _args()
    for call in (lambda: dlm.dlm_guided_accept(*a.values()), lambda: dlm.dlm_guided_accept(**a)):
        with pytest.raises(TypeError, match="contiguous CUDA tensor"):
            call()
    with pytest.raises(ValueError):
        dlm.dlm_guided_accept(None, *([None] * 2), "one", 4, *([None] * 2), 0, *([None] * 3))
    with pytest.raises(TypeError):      # the cache is not a dlm_kv_cache
        dlm.dlm_kv_cache_commit(None, None, None, None, 1, None, None, 0, None, 1, 0, 0, 1)


def test_bytes_of_other_objects_are_not_taken_for_addresses():
    """A context or a cache is what the package makes, not any object with a buffer of that size."""
    other = [b"\0" * 64, bytearray(64), np.zeros(64, np.uint8), (ctypes.c_char * 64)(), ctypes.c_int64(0)]
    for wrong in other:
        with pytest.raises(TypeError, match="expected"):
            dlm.dlm_guided_accept(wrong, None, None, 1, 4, None, None, 0, None, None, None)
    for wrong in other + [ctypes.c_void_p(), 0]:
        with pytest.raises(TypeError, match="expected"):
            dlm.dlm_kv_cache_commit(None, wrong, None, None, 1, None, None, 0, None, 1, 0, 0, 1)
    with pytest.raises(OverflowError):
        dlm.dlm_guided_accept(1 << 70, None, None, 1, 4, None, None, 0, None, None, None)


def test_a_module_for_another_torch_is_stale_and_not_loaded(monkeypatch):
    """The module reads torch's C++ objects: one built for another torch (or Python) is rebuilt however new its file is, and is
    refused before it is loaded."""
    from paper_2505_21467_b200 import _binding
    assert _build.calls_built_for(_build.calls_fingerprint()) and _binding._load_calls().built_for == _build.calls_fingerprint()
    built = []
    monkeypatch.setattr(_build.subprocess, "run", lambda cmd, **kw: built.append(cmd) or _Failed())
    assert _build.build_calls() == _build.CALLS and not built      # fresh: nothing to do
    monkeypatch.setattr(torch, "__version__", "9.9.9")
    with pytest.raises(RuntimeError, match="_dlm_calls"):           # stale: the compiler is called (and fails here)
        _build.build_calls()
    assert len(built) == 1
    monkeypatch.setattr(_binding, "_calls", None)
    with pytest.raises(ImportError, match="not built .* for torch 9.9.9"):
        _binding._load_calls()


def test_a_module_of_other_sources_is_not_loaded(monkeypatch):
    """Nor is one whose functions may be other ones than the package calls: importing the package has to stay possible, or it
    could not be built again."""
    from paper_2505_21467_b200 import _binding
    monkeypatch.setattr(_build, "CALLS_SRC", __file__)
    monkeypatch.setattr(_binding, "_calls", None)
    with pytest.raises(ImportError, match="present sources"):
        _binding._load_calls()
    monkeypatch.setattr(_build, "CALLS_SRC", __file__ + ".not_there")     # a copy of the built package without its sources
    assert _binding._load_calls().built_for
    monkeypatch.setattr(torch, "__version__", "9.9.9")
    monkeypatch.setattr(_binding, "_calls", None)
    with pytest.raises(ImportError, match="torch 9.9.9"):
        _binding._load_calls()


class _Failed:
    returncode, stdout = 1, ""


def test_ctypes_declares_the_calls_that_go_through_it_and_no_others():
    """One declaration per function: the enqueueing calls have theirs in the native module."""
    import re
    from paper_2505_21467_b200 import _binding
    source = open(_binding.__file__).read()
    used = set(re.findall(r"lib\(\)\.(dlm_\w+)", source))
    declared = set(re.findall(r'\("(dlm_\w+)", \S+, \[', source)) | set(re.findall(r"\bL\.(dlm_\w+)\.", source))
    assert declared == used
    assert all(getattr(_binding.lib(), name).argtypes is None for name in dir(_binding._load_calls()) if name.startswith("dlm_"))
