"""Builds libfmm.so in-tree (paper_2203_07673_gb300/_build/) with nvcc for sm_103a.

Each translation unit under csrc/ is compiled in parallel to an object file,
then linked (with the static CUDA runtime) into one shared library exporting
the C ABI declared in include/fmm.h.  The per-call path from PyTorch tensors
(csrc/torch_calls.cpp) is a host-only extension module beside it, built with
g++ against the installed PyTorch.  Rebuilds only what changed.
"""
from __future__ import annotations

import concurrent.futures as cf
import hashlib
import importlib.util
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OUT = os.path.join(PKG, "_build")
LIB = os.path.join(OUT, "libfmm.so")
CALLS = os.path.join(OUT, "fmm_calls.so")

NVCC = os.environ.get("NVCC", "nvcc")
CXX = os.environ.get("CXX", "g++")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
CFLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC",
          "--expt-relaxed-constexpr", f"-I{INCLUDE}", f"-I{CSRC}"]


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _headers_digest():
    h = hashlib.sha1()
    for d in (CSRC, INCLUDE):
        for f in sorted(os.listdir(d)):
            if f.endswith((".cuh", ".h")):
                with open(os.path.join(d, f), "rb") as fh:
                    h.update(f.encode() + fh.read())
    h.update(" ".join(ARCH + CFLAGS).encode())
    return h.hexdigest()


def _compile(src, digest, extra, force):
    obj = os.path.join(OUT, os.path.basename(src)[:-3] + ".o")
    stamp = obj + ".stamp"
    with open(src, "rb") as fh:
        key = digest + hashlib.sha1(fh.read()).hexdigest() + " ".join(extra)
    if not force and os.path.exists(obj) and os.path.exists(stamp):
        if open(stamp).read() == key:
            return obj, False
    cmd = [NVCC, *ARCH, *CFLAGS, *extra, "-c", src, "-o", obj]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{res.stderr}")
    with open(stamp, "w") as fh:
        fh.write(key)
    return obj, True


def _run(cmd, what):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"{cmd[0]} failed for {what}:\n{res.stderr}")


def _drop_calls():
    """Removes the module of the call path (and its stamp)."""
    for path in (CALLS + ".stamp", CALLS):
        if os.path.exists(path):
            os.remove(path)


def _compile_calls(force):
    """Compiles csrc/torch_calls.cpp against the installed PyTorch; returns the
    object file, PyTorch's directory and the key of both, or None where the
    module is up to date.  A module of another key is removed first."""
    src, obj = os.path.join(CSRC, "torch_calls.cpp"), os.path.join(OUT, "torch_calls.o")
    spec = importlib.util.find_spec("torch")
    if spec is None:
        raise RuntimeError("PyTorch is not installed")
    torch_dir = os.path.dirname(spec.origin)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    inc = [INCLUDE, os.path.join(torch_dir, "include"),
           os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    cmd = [CXX, "-O2", "-std=c++17", "-fPIC", *(f"-I{d}" for d in inc), "-c", src, "-o", obj]
    h = hashlib.sha1(" ".join(cmd).encode())
    for path in (src, os.path.join(INCLUDE, "fmm.h"), os.path.join(torch_dir, "version.py")):
        with open(path, "rb") as fh:
            h.update(fh.read())
    stamp = CALLS + ".stamp"   # written once the module is linked
    if not force and os.path.exists(CALLS) and os.path.exists(stamp):
        with open(stamp) as fh:
            if fh.read() == h.hexdigest():
                return None
    _drop_calls()
    _run(cmd, src)
    return obj, torch_dir, h.hexdigest()


def _link_calls(obj, torch_dir, key):
    tmp = CALLS + f".tmp{os.getpid()}"
    _run([CXX, "-shared", obj, "-o", tmp, f"-L{os.path.join(torch_dir, 'lib')}", "-lc10",
          "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python", f"-L{OUT}", "-l:libfmm.so",
          "-Wl,-rpath,$ORIGIN"], CALLS)
    os.replace(tmp, CALLS)
    with open(CALLS + ".stamp", "w") as fh:
        fh.write(key)


def build_library(force: bool = False, extra_flags=(), verbose: bool = False) -> str:
    """Compile and link libfmm.so; returns its path."""
    os.makedirs(OUT, exist_ok=True)
    digest = _headers_digest()
    extra = list(extra_flags)
    with cf.ThreadPoolExecutor(max_workers=max(1, min(8, os.cpu_count() or 1))) as ex:
        calls = ex.submit(_compile_calls, force)
        results = list(ex.map(lambda s: _compile(s, digest, extra, force), sources()))
    objs = [o for o, _ in results]
    changed = any(c for _, c in results)
    if changed or force or not os.path.exists(LIB):
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [NVCC, *ARCH, "-shared", "-o", tmp, *objs]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(f"link failed:\n{res.stderr}")
        os.replace(tmp, LIB)
    try:
        built = calls.result()
        if built is not None:
            _link_calls(*built)
    except (RuntimeError, OSError) as e:
        # every call then takes its path in Python: slower, the same results
        _drop_calls()
        print(f"{CALLS} not built: {e}", file=sys.stderr)
    if verbose:
        print(LIB)
    return LIB


if __name__ == "__main__":
    build_library(force=True, verbose=True)
