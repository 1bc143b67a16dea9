"""Compiles the CUDA sources into the in-tree shared libraries (sm_100a only).

libspecext.so is the product.  libspecext_testing.so is the same code compiled with -DSPECEXT_TESTING
plus the CUDA-core cross-check kernel and a few test hooks (csrc/testing.h); only the tests load it.
_binding.so is the Python extension module that marshals the calls of a decoding step (csrc/binding.cpp).
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB_PATH = os.path.join(HERE, "libspecext.so")
BINDING_PATH = os.path.join(HERE, "_binding.so")
TESTING_LIB_PATH = os.path.join(HERE, "libspecext_testing.so")
SOURCES = ["api.cu", "attn_tc2.cu", "verify.cu", "prefill.cu", "merge.cu", "retrieval.cu"]
TESTING_SOURCES = SOURCES + ["attn_simt.cu", "testing.cu"]


def nvcc_path() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale(lib: str, deps) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = list(deps) + [os.path.join(os.path.dirname(HERE), "include", "specext.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _cuda_deps():
    return [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")]


def needs_build() -> bool:
    return _stale(LIB_PATH, _cuda_deps())


def _run(cmd, lib: str, verbose: bool) -> str:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError(f"{os.path.basename(cmd[0])} failed building {os.path.basename(lib)}")
    return lib


def _compile(lib: str, sources, defines, verbose: bool) -> str:
    cmd = [nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
           "-shared", "-Xcompiler", "-fPIC", "-cudart", "static", "-o", lib] + list(defines)
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in sources]
    return _run(cmd, lib, verbose)


def binding_tag() -> str:
    """What the extension module is compiled against: its code depends on the layout of torch's and Python's objects."""
    import torch
    return f"specext binding for torch {torch.__version__}, {sysconfig.get_config_var('SOABI')}"


def binding_fits(path: str = BINDING_PATH) -> bool:
    """Whether the module at `path` was built against the torch and the Python that run now (it carries its tag)."""
    with open(path, "rb") as f:
        return (binding_tag() + "\0").encode() in f.read()


def build_binding(force: bool = False, verbose: bool = False) -> str:
    """Builds the extension module against the installed torch and returns its path."""
    src = os.path.join(CSRC, "binding.cpp")
    if not force and not _stale(BINDING_PATH, [src]) and binding_fits():
        return BINDING_PATH
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(nvcc_path())) if os.path.isabs(nvcc_path()) else "/usr/local/cuda"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-o", BINDING_PATH, src,
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DSPX_BUILT_FOR="{binding_tag()}"',
           "-I" + sysconfig.get_paths()["include"], "-I" + os.path.join(root, "include"),
           "-I" + os.path.join(root, "include", "torch", "csrc", "api", "include"), "-I" + os.path.join(cuda, "include"),
           "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    return _run(cmd, BINDING_PATH, verbose)


def build(force: bool = False, verbose: bool = False) -> str:
    """Builds libspecext.so, then the extension module, next to this file and returns the library's path."""
    if force or needs_build():
        _compile(LIB_PATH, SOURCES, [], verbose)
    build_binding(force, verbose)
    return LIB_PATH


def build_testing(force: bool = False, verbose: bool = False) -> str:
    """Builds the test library (cross-check kernel and test hooks) and returns its path."""
    if not force and not _stale(TESTING_LIB_PATH, _cuda_deps()):
        return TESTING_LIB_PATH
    return _compile(TESTING_LIB_PATH, TESTING_SOURCES, ["-DSPECEXT_TESTING"], verbose)


def build_all(force: bool = False, verbose: bool = False) -> None:
    """Both libraries, compiled side by side."""
    with ThreadPoolExecutor(2) as ex:
        a = ex.submit(build, force, verbose)
        b = ex.submit(build_testing, force, verbose)
        a.result()
        b.result()


if __name__ == "__main__":
    build_all(force=True, verbose="-v" in sys.argv)
    print(LIB_PATH)
    print(TESTING_LIB_PATH)
