"""Builds the C-ABI CUDA library ``libdlm.so`` in-tree with nvcc for sm_100a, and the Python entry points of its calls
(``_dlm_calls.so``, a CPython module that links it) with g++."""
from __future__ import annotations

import glob
import hashlib
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libdlm.so")
CALLS = os.path.join(HERE, "_dlm_calls.so")
CALLS_SRC = os.path.join(CSRC, "py_calls.cpp")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared", "-Xptxas", "-v",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into libdlm.so (cross-compiles without a GPU)."""
    if not force and not is_stale():
        build_calls(force=False, verbose=verbose)
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [nvcc, *NVCC_FLAGS, "-I", INCLUDE, "-I", CSRC, "-o", tmp, *sources()]
    proc = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if verbose or proc.returncode != 0:
        sys.stderr.write(proc.stdout)
    if proc.returncode != 0:
        raise RuntimeError("nvcc failed building libdlm.so")
    check_attention_registers(proc.stdout)
    os.replace(tmp, LIB)
    build_calls(force=force, verbose=verbose)
    return LIB


def calls_abi() -> str:
    """Whose C++ and C objects _dlm_calls.so reads: this torch's and this Python's."""
    import torch
    return f"torch {torch.__version__} {torch.version.git_version} {sys.implementation.cache_tag}"


def calls_fingerprint() -> str:
    """What _dlm_calls.so is built from and for.  The module carries it (DLM_CALLS_BUILT_FOR), so that one built for another
    torch or another Python counts as stale however new its file is."""
    h = hashlib.sha256()
    for d in [CALLS_SRC, *sorted(glob.glob(os.path.join(INCLUDE, "*.h")))]:
        with open(d, "rb") as f:
            h.update(f.read())
    return f"dlm_calls for {calls_abi()}, sources {h.hexdigest()}"


def calls_built_for(what: str) -> bool:
    """Whether the _dlm_calls.so in place carries `what` (read from the file: a module for another torch is not loaded)."""
    try:
        with open(CALLS, "rb") as f:
            return what.encode() in f.read()
    except OSError:
        return False


def calls_loadable() -> bool:
    """Whether the _dlm_calls.so in place may be loaded: built for this torch and Python and, where the sources are at hand (a
    copy of the built package may come without them), from them."""
    at_hand = os.path.exists(CALLS_SRC) and os.path.exists(os.path.join(INCLUDE, "dlm.h"))
    return calls_built_for(calls_fingerprint() if at_hand else f"dlm_calls for {calls_abi()}, ")


def build_calls(force: bool = False, verbose: bool = False) -> str:
    """Compile the Python entry points (needs torch's headers, no GPU)."""
    if not force and calls_built_for(calls_fingerprint()):
        return CALLS
    import torch
    from torch.utils import cpp_extension
    tmp = CALLS + f".{os.getpid()}.tmp"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           f'-DDLM_CALLS_BUILT_FOR="{calls_fingerprint()}"',
           "-I", INCLUDE, "-I", sysconfig.get_paths()["include"]]
    for d in cpp_extension.include_paths("cuda"):
        cmd += ["-isystem", d]
    cmd += ["-o", tmp, CALLS_SRC, "-L", HERE, "-l:libdlm.so", "-Wl,-rpath,$ORIGIN"]
    for d in cpp_extension.library_paths("cuda"):
        cmd += ["-L", d]
    cmd += ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    proc = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if verbose or proc.returncode != 0:
        sys.stderr.write(proc.stdout)
    if proc.returncode != 0:
        raise RuntimeError("g++ failed building _dlm_calls.so")
    os.replace(tmp, CALLS)
    return CALLS


# The attention kernel moves registers between its warpgroups with setmaxnreg: 8 softmax warps grow to 216 registers a
# thread from what the other 4 warps give up when they shrink to 72, which balances only if the kernel is launched
# with 168 (attn_step.cu: kRegsSoftmax, kRegsOther, register_budget_ok).  A compiler that allocates another number
# would make every attention call fail at run time with DLM_ERR_UNSUPPORTED; fail the build instead.
ATTENTION_REGISTERS = 168


def check_attention_registers(ptxas_log: str) -> None:
    seen, name = 0, None
    for line in ptxas_log.splitlines():
        if "Compiling entry function" in line:
            name = line.split("'")[1] if "'" in line else line
        elif "Used" in line and "registers" in line and name is not None:
            if "attn_step_sm100_kernel" in name:
                seen += 1
                regs = int(line.split("Used")[1].split("registers")[0])
                if regs != ATTENTION_REGISTERS:
                    raise RuntimeError(f"{name}: ptxas allocated {regs} registers, the kernel's register split needs "
                                       f"{ATTENTION_REGISTERS}")
            name = None
    if seen == 0:
        raise RuntimeError("no attention kernel found in the ptxas log: cannot check its register count")


if __name__ == "__main__":
    build(force=True, verbose=True)
    print(LIB)
