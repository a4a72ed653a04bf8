"""Build libsph.so (the C-ABI library) from csrc/ with nvcc for sm_103a.

Each translation unit compiles in parallel to an object file under _lib/;
the objects link into _lib/libsph.so against the shared CUDA runtime (the
same libcudart the process already uses for PyTorch).  A source newer than
its object, or a changed header, triggers a rebuild of that unit.  The library
needs nvcc alone.  Where PyTorch is installed, nvcc's host compiler builds the
binding's native argument marshalling beside it, in a file that carries the
PyTorch and Python it was built against in its name (fast_path): another
PyTorch or Python never loads it.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OUT = os.path.join(PKG, "_lib")
LIB = os.path.join(OUT, "libsph.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC",
              "--expt-relaxed-constexpr", "-Xptxas", "-warn-spills"]


def nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _headers():
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC)
          if f.endswith((".h", ".cuh"))]
    hs += [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE) if f.endswith(".h")]
    return hs


def _stale(obj: str, src: str, newest_header: float) -> bool:
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    return os.path.getmtime(src) > t or newest_header > t


def fast_path():
    """File of the native argument marshalling for the running Python and the
    installed PyTorch; None without PyTorch."""
    try:
        import torch
    except ImportError:
        return None
    abi = sysconfig.get_config_var("SOABI")
    return os.path.join(OUT, f"py_fast.{abi}.torch-{torch.__version__}.so")


def _fast_cmd(cc: str, src: str, out: str):
    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    inc, lib = os.path.join(root, "include"), os.path.join(root, "lib")
    abi = int(getattr(torch._C, "_GLIBCXX_USE_CXX11_ABI", True))
    return [cc, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-cudart", "none",
            f"-D_GLIBCXX_USE_CXX11_ABI={abi}", "-I", INCLUDE,
            "-I", sysconfig.get_paths()["include"], "-I", inc,
            "-I", os.path.join(inc, "torch", "csrc", "api", "include"), src, "-o", out,
            "-L", lib, "-Xlinker", f"-rpath={lib}", "-lc10", "-ltorch_cpu", "-ltorch_python", "-ldl"]


def build(verbose: bool = False, force: bool = False, extra_flags=()) -> str:
    """Compile every csrc/*.cu and link _lib/libsph.so, and build the native
    marshalling where PyTorch is installed; returns the library's path."""
    os.makedirs(OUT, exist_ok=True)
    cc = nvcc()
    srcs = _sources()
    newest_header = max(os.path.getmtime(h) for h in _headers())
    objs = []
    jobs = []
    for s in srcs:
        o = os.path.join(OUT, os.path.splitext(os.path.basename(s))[0] + ".o")
        objs.append(o)
        if force or _stale(o, s, newest_header):
            cmd = [cc, *ARCH, *NVCC_FLAGS, *extra_flags, "-I", INCLUDE,
                   "-I", CSRC, "-c", s, "-o", o]
            jobs.append((s, cmd))

    relink = bool(jobs) or force or not os.path.exists(LIB)
    fast, fast_src = fast_path(), os.path.join(CSRC, "py_fast.cpp")
    newest = max(newest_header, os.path.getmtime(os.path.abspath(__file__)))
    if fast and (force or _stale(fast, fast_src, newest)):
        jobs.append((fast_src, _fast_cmd(cc, fast_src, fast)))

    def run(job):
        src, cmd = job
        if verbose:
            print(" ".join(cmd), flush=True)
        r = subprocess.run(cmd, capture_output=True, text=True)
        return src, r

    failed = []
    with cf.ThreadPoolExecutor(max_workers=max(1, min(len(jobs), os.cpu_count() or 4))) as ex:
        for src, r in ex.map(run, jobs):
            if verbose and (r.stdout or r.stderr):
                print(r.stdout + r.stderr, flush=True)
            if r.returncode != 0:
                failed.append((src, r.stdout + r.stderr))
    if relink and not any(s != fast_src for s, _ in failed):
        cmd = [cc, *ARCH, "-shared", "-cudart", "shared", "-o", LIB, *objs]
        if verbose:
            print(" ".join(cmd), flush=True)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("link failed:\n" + r.stdout + r.stderr)
    if failed:          # (the marshalling's failure leaves the library linked)
        msg = "\n".join(f"{s}:\n{out}" for s, out in failed)
        raise RuntimeError("compiling failed:\n" + msg)
    return LIB


if __name__ == "__main__":
    print(build(verbose=True, force="--force" in sys.argv))
