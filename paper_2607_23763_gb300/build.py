"""In-tree build of libsosfilt.so for sm_103a (nvcc only, no cmake).

Each translation unit is compiled in its own nvcc process (in parallel), then
linked into ``paper_2607_23763_gb300/libsosfilt.so``.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
ROOT = os.path.dirname(PKG)
OUT = os.path.join(PKG, "libsosfilt.so")
NATIVE_SRC = os.path.join(CSRC, "py", "native.cpp")
NATIVE = os.path.join(PKG, "_native.so")
OBJ = os.path.join(PKG, "_build")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
COMMON = ["-std=c++17", "-O3", "-lineinfo", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include")]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA library cannot be built")


def sources() -> list[str]:
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cpp")))


def build_native(force: bool = False) -> None:
    """The binding's argument marshalling (csrc/py/native.cpp), an extension module against the installed
    torch.  Without it (no headers or no torch here) the binding marshals in Python."""
    if not force and not _stale(NATIVE, [NATIVE_SRC]):
        return
    try:
        import sysconfig

        import torch
        root = os.path.dirname(torch.__file__)
        cuda = os.path.dirname(os.path.dirname(_nvcc()))
        tmp = f"{NATIVE}.{os.getpid()}.tmp"
        subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-o", tmp, NATIVE_SRC,
                        "-I", sysconfig.get_paths()["include"], "-I", os.path.join(root, "include"),
                        "-I", os.path.join(root, "include", "torch", "csrc", "api", "include"),
                        "-I", os.path.join(cuda, "include"), f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                        "-L", os.path.join(root, "lib"), f"-Wl,-rpath,{os.path.join(root, 'lib')}",
                        "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"],
                       check=True, capture_output=True, text=True)
        os.replace(tmp, NATIVE)
    except (ImportError, OSError, subprocess.CalledProcessError) as e:
        sys.stderr.write(f"the binding's native marshalling was not built: {getattr(e, 'stderr', e)}\n")


def _stale(out: str, deps: list[str]) -> bool:
    if not os.path.exists(out):
        return True
    t = os.path.getmtime(out)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    nvcc = _nvcc()
    os.makedirs(OBJ, exist_ok=True)
    srcs = sources()
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    headers.append(os.path.join(ROOT, "include", "sosfilt.h"))
    jobs = []
    for src in srcs:
        obj = os.path.join(OBJ, os.path.basename(src) + ".o")
        if force or _stale(obj, [src] + headers):
            lang = ["-x", "cu"] if src.endswith(".cu") else ["-x", "c++"]
            jobs.append([nvcc, *COMMON, *ARCH, *lang, "-c", src, "-o", obj])
    native = cf.ThreadPoolExecutor(max_workers=1)
    native_done = native.submit(build_native, force)
    if jobs:
        with cf.ThreadPoolExecutor(max_workers=min(len(jobs), os.cpu_count() or 4)) as ex:
            results = list(ex.map(lambda c: subprocess.run(c, capture_output=True, text=True), jobs))
        for cmd, res in zip(jobs, results):
            if verbose or res.returncode:
                sys.stderr.write(" ".join(cmd) + "\n" + res.stdout + res.stderr)
            if res.returncode:
                raise RuntimeError(f"nvcc failed on {cmd[-3]}")
    native_done.result()
    native.shutdown()
    objs = [os.path.join(OBJ, os.path.basename(s) + ".o") for s in srcs]
    if force or jobs or _stale(OUT, objs):
        tmp = f"{OUT}.{os.getpid()}.tmp"
        cmd = [nvcc, *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode:
            raise RuntimeError("link failed:\n" + res.stdout + res.stderr)
        os.replace(tmp, OUT)
    return OUT


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
