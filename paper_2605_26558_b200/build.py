"""In-tree build of the CUDA library (sm_100a only) with nvcc and of its CPython entry points with g++; no torch extension machinery."""
from __future__ import annotations

import concurrent.futures
import importlib.metadata
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcass.so")
FASTCALL = os.path.join(HERE, "_fastcall.so")          # CPython entry points of the library (csrc/fastcall.cpp)
FASTCALL_FOR = os.path.join(HERE, "_build", "_fastcall.txt")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
         "--expt-relaxed-constexpr"]


def sources() -> list[str]:
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _stale(target: str, deps: list[str]) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _fastcall_for() -> str:
    """What the entry points are compiled against: another torch or interpreter may lay its objects out otherwise."""
    return f"torch {importlib.metadata.version('torch')} {sys.implementation.cache_tag}"


def _fastcall_current(src: str, header: str) -> bool:
    if _stale(FASTCALL, [src, header]) or not os.path.exists(FASTCALL_FOR):
        return False
    with open(FASTCALL_FOR) as f:
        return f.read() == _fastcall_for()


def _build_fastcall(header: str, force: bool) -> None:
    src = os.path.join(CSRC, "fastcall.cpp")
    if not force and _fastcall_current(src, header):
        return
    import sysconfig

    import torch

    troot = os.path.dirname(torch.__file__)
    inc = [os.path.join(troot, "include"), os.path.join(troot, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include")]
    cmd = (["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"] +
           [f"-I{i}" for i in inc] + [src, "-o", FASTCALL, "-L" + HERE, "-l:libcass.so", "-L" + os.path.join(troot, "lib"), "-ltorch_python", "-ltorch_cpu",
                                     "-ltorch", "-lc10", "-lc10_cuda", "-Wl,-rpath,$ORIGIN"])
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed for {src}:\n{r.stdout}\n{r.stderr}")
    with open(FASTCALL_FOR, "w") as f:
        f.write(_fastcall_for())


def build(force: bool = False, verbose: bool = False) -> str:
    srcs = sources()
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(os.path.dirname(HERE), "include", "cass.h"))
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    jobs = []
    for s in srcs:
        o = os.path.join(objdir, os.path.basename(s)[:-3] + ".o")
        if force or _stale(o, [s] + headers):
            jobs.append((s, o))

    def compile_one(job):
        s, o = job
        cmd = [NVCC] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", s, "-o", o]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {s}:\n{r.stdout}\n{r.stderr}")
        return r.stderr

    with concurrent.futures.ThreadPoolExecutor(max_workers=8) as ex:
        for log in ex.map(compile_one, jobs):
            if verbose and log:
                print(log, file=sys.stderr)
    objs = [os.path.join(objdir, os.path.basename(s)[:-3] + ".o") for s in srcs]
    if force or jobs or _stale(LIB, objs):
        cmd = [NVCC, "-shared", "-o", LIB] + objs + ["-lcudart"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    _build_fastcall(os.path.join(os.path.dirname(HERE), "include", "cass.h"), force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
