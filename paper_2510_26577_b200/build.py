"""Builds the CAST CUDA library in-tree: csrc/*.cu -> libcast_b200.so (sm_100a only), and the native side of the
Python binding: csrc/binding_calls.cpp -> _cast_calls.so."""
from __future__ import annotations

import importlib.util
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(ROOT, "build", "obj")
LIB = os.path.join(PKG, "libcast_b200.so")
CALLS = os.path.join(PKG, "_cast_calls.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _built_against(torch_dir: str) -> str:
    """What the extension module is good for: this torch (its classes are linked to by mangled name) and this Python."""
    with open(os.path.join(torch_dir, "version.py")) as f:
        return (sysconfig.get_config_var("SOABI") or sys.version) + "\n" + torch_dir + "\n" + f.read()


def _build_calls() -> None:
    """The extension module the binding calls through (host code against torch's headers; links the CUDA library)."""
    src = os.path.join(CSRC, "binding_calls.cpp")
    torch_dir = os.path.dirname(importlib.util.find_spec("torch").origin)
    stamp, against = os.path.join(OBJ, "binding_calls.against"), _built_against(torch_dir)
    same = False
    if os.path.exists(stamp):
        with open(stamp) as f:
            same = f.read() == against
    if same and not _stale(CALLS, [src, os.path.join(ROOT, "include", "cast.h"), os.path.abspath(__file__)]):
        return
    inc, lib = os.path.join(torch_dir, "include"), os.path.join(torch_dir, "lib")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    cmd = ["g++", "-shared", "-fPIC", "-O2", "-std=c++17", "-fvisibility=hidden", "-I", os.path.join(ROOT, "include"),
           "-I", inc, "-I", os.path.join(inc, "torch", "csrc", "api", "include"), "-I", cuda,
           "-I", sysconfig.get_paths()["include"], src, "-o", CALLS, "-L", lib, "-lc10", "-lc10_cuda", "-ltorch_cpu",
           "-ltorch_python", "-L", PKG, "-lcast_b200", "-Wl,-rpath,$ORIGIN"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        raise RuntimeError("g++ failed for binding_calls.cpp")
    with open(stamp, "w") as f:
        f.write(against)


def build(verbose: bool = False, force: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    sources = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".h")]
    headers.append(os.path.join(ROOT, "include", "cast.h"))
    headers.append(os.path.abspath(__file__))
    jobs = []
    objs = []
    for src in sources:
        s = os.path.join(CSRC, src)
        o = os.path.join(OBJ, src[:-3] + ".o")
        objs.append(o)
        if force or _stale(o, [s] + headers):
            cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", s, "-o", o]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        return cmd, r

    with ThreadPoolExecutor(max_workers=min(8, max(1, len(jobs)))) as ex:
        for cmd, r in ex.map(run, jobs):
            if verbose or r.returncode != 0:
                sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr + "\n")
            if r.returncode != 0:
                raise RuntimeError("nvcc failed for " + cmd[-3])
    if jobs or force or _stale(LIB, objs):
        cmd = [_nvcc(), "-shared", "-o", LIB] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
    _build_calls()
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, force="-f" in sys.argv))
