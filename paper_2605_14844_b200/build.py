"""Build libxfp.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and the binding's native marshalling module."""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(CSRC, "build" + ("_" + os.environ["XFP_LIBTAG"] if os.environ.get("XFP_LIBTAG") else ""))
# XFP_LIBTAG=name builds libxfp_name.so from objects of its own (csrc/build_name), with the extra -D flags of
# XFP_DEFS: a way to keep several builds side by side when comparing kernel variants
TAG = os.environ.get("XFP_LIBTAG", "")
LIB = os.path.join(HERE, f"libxfp_{TAG}.so" if TAG else "libxfp.so")
NATIVE = os.path.join(HERE, "_xfp_native.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-Xptxas", "-v"]
# XFP_TRACE=1 compiles the per-CTA phase stamps of the pair kernel in (a timing probe; use with --force)
if os.environ.get("XFP_TRACE") == "1":
    FLAGS.append("-DXFP_TRACE=1")
FLAGS += [f"-D{d}" for d in os.environ.get("XFP_DEFS", "").split()]


def _sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _headers_mtime():
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    inc = os.path.join(HERE, "..", "include")
    hs += [os.path.join(inc, f) for f in os.listdir(inc) if f.endswith(".h")]
    return max(os.path.getmtime(h) for h in hs)


def _build_native(force: bool) -> None:
    """_xfp_native.so, the marshalling module of the Python binding (g++ against torch's headers)."""
    import sysconfig
    import torch
    src = os.path.join(CSRC, "xfp_native.cpp")
    if not force and os.path.exists(NATIVE) and os.path.getmtime(NATIVE) >= max(os.path.getmtime(src), _headers_mtime()):
        return
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(NVCC))
    inc = [sysconfig.get_paths()["include"], os.path.join(root, "include"),
           os.path.join(root, "include", "torch", "csrc", "api", "include"), os.path.join(cuda, "include")]
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++20", "-fPIC", "-shared", "-w",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *[f"-I{i}" for i in inc], src, "-o", NATIVE + ".tmp",
           f"-L{os.path.join(root, 'lib')}", "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode:
        raise RuntimeError(f"g++ failed on {src}:\n{r.stdout}\n{r.stderr}")
    os.replace(NATIVE + ".tmp", NATIVE)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    hm = _headers_mtime()
    jobs = []
    for src in _sources():
        s = os.path.join(CSRC, src)
        o = os.path.join(OBJ, src[:-3] + ".o")
        if force or not os.path.exists(o) or os.path.getmtime(o) < max(os.path.getmtime(s), hm):
            jobs.append((s, o))

    def compile_one(job):
        s, o = job
        r = subprocess.run([NVCC, *FLAGS, "-c", s, "-o", o], capture_output=True, text=True)
        with open(o + ".log", "w") as f:
            f.write(r.stdout + r.stderr)
        if r.returncode:
            raise RuntimeError(f"nvcc failed on {s}:\n{r.stdout}\n{r.stderr}")
        if verbose:
            sys.stderr.write(r.stderr)
        return o

    with ThreadPoolExecutor(max_workers=8) as ex:
        native = ex.submit(_build_native, force)
        list(ex.map(compile_one, jobs))
        native.result()
    objs = [os.path.join(OBJ, src[:-3] + ".o") for src in _sources()]
    if jobs or not os.path.exists(LIB):
        r = subprocess.run([NVCC, "-shared", "-o", LIB + ".tmp", *objs], capture_output=True, text=True)
        if r.returncode:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
        os.replace(LIB + ".tmp", LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
