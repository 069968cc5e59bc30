"""Builds ``libspec_attn.so`` (nvcc, sm_100a) and ``_spec_native.so`` (g++, the argument marshalling of
binding.py) in-tree; cross-compiles without a GPU.

``python -m paper_2607_27735_b200.build [--force] [--verbose]``
"""
from __future__ import annotations

import concurrent.futures
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "build")
LIB = os.path.join(HERE, "libspec_attn.so")
NATIVE = os.path.join(HERE, "_spec_native.so")
NATIVE_SRC = os.path.join(CSRC, "py_native.cpp")
SOURCES = ["spec_api.cu", "verify_generic.cu", "verify_sm100.cu", "verify_sm100_twosweep.cu",
           "verify_sm100_cached.cu", "verify_sm100_cached_rows.cu", "verify_sm100_cached_ph.cu", "verify_sm100_cached_ph_rows.cu",
           "verify_sm100_cached_sc.cu", "verify_sm100_cached_f8.cu", "select_recall.cu", "draft_stream.cu", "spec_noalloc.cu",
           "length_ctrl.cu", "kv_expand.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
              "-I", CSRC]


def _newest_dep() -> float:
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")]
    deps.append(os.path.join(ROOT, "include", "spec_attn.h"))
    return max(os.path.getmtime(p) for p in deps)


def _compile(src: str, verbose: bool) -> str:
    obj = os.path.join(OBJ, src.replace(".cu", ".o"))
    cmd = ["nvcc", *NVCC_FLAGS, *os.environ.get("SPEC_EXTRA_NVCC_FLAGS", "").split(), "-c",
           os.path.join(CSRC, src), "-o", obj]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}")
    return obj


def native_abi() -> str:
    """What the Python module is compiled against, as text the module carries: it uses torch's C++ interface, so a
    module built beside another torch or interpreter must not be loaded."""
    import torch

    return f"torch {torch.__version__} python {sys.version_info[0]}.{sys.version_info[1]}"


def _native_current() -> bool:
    """Whether the built module is newer than its sources and compiled against this torch and interpreter."""
    if not os.path.exists(NATIVE) or os.path.getmtime(NATIVE) < max(
            os.path.getmtime(NATIVE_SRC), os.path.getmtime(os.path.join(ROOT, "include", "spec_attn.h"))):
        return False
    with open(NATIVE, "rb") as f:
        return native_abi().encode() + b"\0" in f.read()


def _native_obj(verbose: bool) -> str:
    """Object file of the Python module (torch's headers make it the slowest host file: compiled beside the kernels)."""
    import torch
    from torch.utils import cpp_extension

    obj = os.path.join(OBJ, "py_native.o")
    inc = [*cpp_extension.include_paths(), sysconfig.get_paths()["include"], os.path.join(ROOT, "include"),
           os.path.join(cpp_extension.CUDA_HOME or "/usr/local/cuda", "include")]
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           f'-DSPEC_NATIVE_ABI="{native_abi()}"', *(f"-I{p}" for p in inc), "-c", NATIVE_SRC, "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError("g++ failed on py_native.cpp")
    return obj


def _link_native(obj: str) -> None:
    import torch

    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    # libspec_attn.so is found next to the module; torch's libraries are loaded by the time it is imported
    subprocess.check_call(["g++", "-shared", "-o", NATIVE, obj, LIB, f"-L{lib}", "-ltorch_python", "-ltorch_cpu", "-lc10",
                           "-lc10_cuda", "-Wl,-rpath,$ORIGIN"])


def build(force: bool = False, verbose: bool = False) -> str:
    lib_old = force or not os.path.exists(LIB) or os.path.getmtime(LIB) < _newest_dep()
    native_old = force or not _native_current()
    os.makedirs(OBJ, exist_ok=True)
    with concurrent.futures.ThreadPoolExecutor(max_workers=len(SOURCES) + 1) as ex:
        native = ex.submit(_native_obj, verbose) if native_old else None
        if lib_old:
            objs = list(ex.map(lambda s: _compile(s, verbose), SOURCES))
            subprocess.check_call(["nvcc", "-shared", "-Wno-deprecated-gpu-targets", "-o", LIB, *objs, "-cudart", "static",
                                   "-Xlinker", "-soname=libspec_attn.so"])
        if native is not None:
            _link_native(native.result())
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
