"""Builds libcachespec.so in-tree for sm_103a (nvcc, one -gencode, parallel TUs)
and the binding's marshalling module beside it (g++, against the installed torch).

``python -m paper_2607_20507_gb300.build [--force] [--ptxas-v]``
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
INCLUDE = os.path.join(ROOT, "include")
BUILD_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libcachespec.so")
MARSHAL = os.path.join(HERE, "_marshal.so")
AGAINST = os.path.join(BUILD_DIR, "marshal.against")
SOURCES = ["capi.cu", "verify_attention.cu", "spec_accept.cu", "noalloc.cu", "kv_cache.cu", "route.cu", "selftest.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _inputs() -> list[str]:
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files += [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    files.append(os.path.abspath(__file__))
    return files


def _built_against() -> str:
    """What the marshalling module's binary interface comes from."""
    import torch
    return f"python {sys.version}\ntorch {torch.__version__} {os.path.dirname(torch.__file__)}\n"


def is_stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(MARSHAL) or not os.path.exists(AGAINST):
        return True
    with open(AGAINST) as f:
        if f.read() != _built_against():
            return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(MARSHAL))
    return any(os.path.getmtime(f) > t for f in _inputs())


def _run(cmd: list[str], what: str) -> str:
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"{what} failed:\n{r.stdout}\n{r.stderr}")
    return r.stdout + r.stderr


def _compile_marshal() -> str:
    import torch
    home = os.path.dirname(torch.__file__)
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    obj = os.path.join(BUILD_DIR, "marshal.o")
    _run(["g++", "-O2", "-std=c++17", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
          "-I", INCLUDE, "-I", os.path.join(home, "include"),
          "-I", os.path.join(home, "include", "torch", "csrc", "api", "include"),
          "-I", sysconfig.get_paths()["include"], "-I", cuda,
          "-c", os.path.join(CSRC, "marshal.cpp"), "-o", obj], "g++ marshal.cpp")
    return obj


def _link_marshal(obj: str) -> None:
    import torch
    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = MARSHAL + f".tmp{os.getpid()}"
    _run(["g++", "-shared", "-o", tmp, obj, "-L", libs, "-L", HERE, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10",
          "-lc10_cuda", "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + libs], "marshal link")
    os.replace(tmp, MARSHAL)
    with open(AGAINST, "w") as f:
        f.write(_built_against())


def build(force: bool = False, ptxas_verbose: bool = False, quiet: bool = True) -> str:
    if not force and not is_stale():
        return LIB
    os.makedirs(BUILD_DIR, exist_ok=True)
    flags = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC,
             *ARCH]
    if ptxas_verbose:
        flags += ["-Xptxas", "-v"]

    def compile_one(src: str) -> tuple[str, str]:
        obj = os.path.join(BUILD_DIR, src.replace(".cu", ".o"))
        cmd = [_nvcc(), *flags, "-c", os.path.join(CSRC, src), "-o", obj]
        return obj, _run(cmd, f"nvcc {src}")

    with concurrent.futures.ThreadPoolExecutor(max_workers=len(SOURCES) + 1) as ex:
        marshal = ex.submit(_compile_marshal)
        results = list(ex.map(compile_one, SOURCES))
    if ptxas_verbose or not quiet:
        for _, log in results:
            if log.strip():
                print(log, file=sys.stderr)
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [_nvcc(), "-shared", *ARCH, "-o", tmp, *[o for o, _ in results]]
    _run(cmd, "link")
    os.replace(tmp, LIB)
    _link_marshal(marshal.result())
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, ptxas_verbose="--ptxas-v" in sys.argv, quiet=False)
    print(LIB)
