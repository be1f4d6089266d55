"""Builds in-tree: the CUDA library ``libpulsar.so`` (sm_100a only) and ``_native.so``, the native half of the binding."""
from __future__ import annotations

import importlib.metadata
import os
import subprocess
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libpulsar.so")
NATIVE = os.path.join(HERE, "_native.so")
NATIVE_SOURCE = os.path.join(CSRC, "binding.cpp")
NATIVE_KEY = os.path.join(HERE, "build", "_native.key")     # what NATIVE was compiled against
SOURCES = ["api.cu", "select.cu", "merge.cu", "attn.cu", "decode.cu", "rope.cu"]
HEADERS = [os.path.join(CSRC, "common.cuh"), os.path.join(CSRC, "decode.cuh"), os.path.join(os.path.dirname(HERE), "include", "pulsar.h")]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale(target: str, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def needs_build() -> bool:
    return _stale(LIB, [os.path.join(CSRC, s) for s in SOURCES] + HEADERS)


def native_key() -> str:
    """The Python and the torch that a build of the extension module is good for: it uses the ABI of both."""
    return f"{sysconfig.get_config_var('SOABI')} torch-{importlib.metadata.version('torch')}"


def _native_stale() -> bool:
    if _stale(NATIVE, [NATIVE_SOURCE, HEADERS[-1]]) or not os.path.exists(NATIVE_KEY):
        return True
    with open(NATIVE_KEY) as f:
        return f.read() != native_key()


def build_native(force: bool = False) -> str:
    """Compile the binding's extension module against the torch that is installed.  Returns its path."""
    if not force and not _native_stale():
        return NATIVE
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    tmp = NATIVE + f".tmp{os.getpid()}"
    subprocess.check_call([
        "g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
        f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
        "-I" + os.path.join(root, "include"), "-I" + os.path.join(root, "include", "torch", "csrc", "api", "include"),
        "-I" + sysconfig.get_path("include"), "-I" + os.path.join(cuda, "include"), NATIVE_SOURCE, "-o", tmp,
        "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"])
    os.replace(tmp, NATIVE)
    os.makedirs(os.path.dirname(NATIVE_KEY), exist_ok=True)
    with open(NATIVE_KEY, "w") as f:
        f.write(native_key())
    return NATIVE


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu for sm_100a and link the shared library, and the binding's module.  Returns the library's path."""
    build_native(force)
    if not force and not needs_build():
        return LIB
    objs = []
    build_dir = os.path.join(HERE, "build")
    os.makedirs(build_dir, exist_ok=True)
    procs = []
    for src in SOURCES:
        obj = os.path.join(build_dir, src.replace(".cu", ".o"))
        cmd = [_nvcc(), *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            print(out)
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.check_call([_nvcc(), "-shared", "-o", tmp, *objs, "-lcudart"])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
