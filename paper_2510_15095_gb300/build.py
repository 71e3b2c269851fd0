"""Builds libhive_gb300.so in-tree with nvcc for sm_103a (GB300), and the
native call path of the Python binding (hive_binding.so) with g++.

The translation units compile in parallel: the kernels (CUDA), the host
library (C++ using the CUDA runtime, linked statically) and the binding, which
uses the installed torch's headers.  The binding is optional (the Python code
makes every call without it, by ctypes): where it does not compile, build()
says so and goes on.
"""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OUT_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(OUT_DIR, "libhive_gb300.so")
SOURCES = ["hive_kernels.cu", "hive32_kernels.cu", "hive_host.cpp", "hive32.cpp", "hive_multi.cpp",
           "hive_hostio.cpp", "hive_vmm.cpp", "hive_contract.cpp", "hive_noalloc.cu"]
HEADERS = ["hive_internal.h", "hive_device.cuh", "hive_tags.cuh"]
BINDING = os.path.join(OUT_DIR, "hive_binding.so")
BINDING_STAMP = os.path.join(OUT_DIR, "hive_binding.built_for")
BINDING_SRC = "hive_binding.cpp"
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _older(path: str, sources) -> bool:
    if not os.path.exists(path):
        return True
    t = os.path.getmtime(path)
    deps = [os.path.join(CSRC, f) for f in sources]
    deps.append(os.path.join(ROOT, "include", "hive.h"))
    deps.append(os.path.abspath(__file__))
    return any(os.path.getmtime(d) > t for d in deps)


def _stale() -> bool:
    return _older(LIB, SOURCES + HEADERS)


def binding_key() -> str:
    """What a built binding depends on besides its source: torch and Python."""
    import importlib.metadata

    try:
        version = importlib.metadata.version("torch")
    except importlib.metadata.PackageNotFoundError:
        import torch

        version = torch.__version__
    return f"torch {version} {sys.implementation.cache_tag}"


def binding_fits() -> bool:
    """Whether the built binding belongs to this torch and Python."""
    try:
        with open(BINDING_STAMP) as f:
            return os.path.exists(BINDING) and f.read() == binding_key()
    except OSError:
        return False


def build_binding() -> str:
    """hive_binding.so: a CPython module compiled against the installed torch."""
    import sysconfig

    import torch

    base = os.path.dirname(torch.__file__)
    inc = os.path.join(base, "include")
    lib = os.path.join(base, "lib")
    cuda = os.path.dirname(os.path.dirname(nvcc())) if os.sep in nvcc() else "/usr/local/cuda"
    tmp = BINDING + f".{os.getpid()}.tmp"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
           "-I", os.path.join(ROOT, "include"), "-isystem", inc,
           "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"),
           "-isystem", os.path.join(cuda, "include"),
           "-isystem", sysconfig.get_paths()["include"],
           os.path.join(CSRC, BINDING_SRC), "-o", tmp, "-L", lib,
           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", f"-Wl,-rpath,{lib}"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed for {BINDING_SRC}:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, BINDING)
    with open(BINDING_STAMP, "w") as f:
        f.write(binding_key())
    return BINDING


def _build_binding() -> None:
    try:
        build_binding()
    except Exception as e:  # noqa: BLE001  (no torch headers, no compiler, ...)
        sys.stderr.write(f"hive_binding.so was not built, calls go through ctypes: {e}\n")


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    lib = force or _stale()
    binding = force or _older(BINDING, [BINDING_SRC]) or not binding_fits()
    os.makedirs(OUT_DIR, exist_ok=True)
    if not lib:
        if binding:
            _build_binding()
        return LIB
    common = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
              "-I", CSRC, *extra_flags]

    def compile_one(src):
        obj = os.path.join(OUT_DIR, os.path.splitext(src)[0] + ".o")
        cmd = [nvcc(), *ARCH, *common, "-c", os.path.join(CSRC, src), "-o", obj]
        if src.endswith(".cu"):
            cmd[1:1] = ["-Xptxas", "-v"] if verbose else []
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        if verbose and r.stderr:
            sys.stderr.write(r.stderr)
        return obj

    with ThreadPoolExecutor(len(SOURCES) + 1) as ex:
        if binding:
            ex.submit(_build_binding)
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [nvcc(), *ARCH, "-shared", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
