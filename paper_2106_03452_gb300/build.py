"""Build libdpsr.so in-tree with nvcc for sm_103a (GB300), and the PyTorch
binding of its hot calls with g++.

Each .cu translation unit is compiled in parallel, then linked into
paper_2106_03452_gb300/_build/libdpsr.so (no torch, no cmake);
csrc/torch_bind.cpp becomes _build/_dpsr_torch.so next to it, against the
headers of the installed PyTorch.
"""
from __future__ import annotations

import concurrent.futures as cf
import hashlib
import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "libdpsr.so")
# the debug build (bounds checks on data-dependent indices, DPSR_DEBUG_CHECKS)
BUILD_DEBUG = os.path.join(HERE, "_build_debug")
LIB_DEBUG = os.path.join(BUILD_DEBUG, "libdpsr.so")
BIND = "torch_bind.cpp"
BIND_NAME = "_dpsr_torch.so"
SOURCES = ["dpsr_api.cu", "k_plane.cu", "k_xpass.cu", "k_points.cu", "k_pencil.cu", "dpsr_static.cu", "dpsr_batch.cu", "dpsr_serve.cu", "k_mesh.cu", "k_opt.cu", "k_chamfer.cu", "tune_cache.cu", "k_peak.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
         "--expt-relaxed-constexpr", "-I", INCLUDE, "-I", CSRC]


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libdpsr")


def _torch():
    import torch
    return torch


def _bind_flags():
    """(compile, link) flags of the binding: PyTorch's headers and libraries."""
    torch = os.path.dirname(_torch().__file__)
    inc = [os.path.join(torch, "include"), os.path.join(torch, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include"),
           INCLUDE]
    abi = f"-D_GLIBCXX_USE_CXX11_ABI={int(_torch().compiled_with_cxx11_abi())}"
    comp = ["-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden", abi, *(f"-I{d}" for d in inc)]
    link = [f"-L{os.path.join(torch, 'lib')}", "-lc10", "-lc10_cuda", "-ltorch", "-ltorch_cpu", "-ltorch_cuda",
            "-ltorch_python", "-ldpsr", "-Wl,-rpath,$ORIGIN"]
    return comp, link


def _fingerprint(extra=()) -> str:
    h = hashlib.sha256()
    for d, names in ((CSRC, sorted(os.listdir(CSRC))), (INCLUDE, sorted(os.listdir(INCLUDE)))):
        for n in names:
            p = os.path.join(d, n)
            if os.path.isfile(p):
                h.update(n.encode())
                with open(p, "rb") as f:
                    h.update(f.read())
    h.update(" ".join(ARCH + FLAGS + list(extra)).encode())
    h.update(f"{_torch().__version__} {sysconfig.get_paths()['include']}".encode())
    return h.hexdigest()


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    """Compile libdpsr.so; with debug=True the bounds-checking variant
    (-DDPSR_DEBUG_CHECKS) into its own folder."""
    build_dir, lib = (BUILD_DEBUG, LIB_DEBUG) if debug else (BUILD, LIB)
    extra = ["-DDPSR_DEBUG_CHECKS=1"] if debug else []
    os.makedirs(build_dir, exist_ok=True)
    stamp = os.path.join(build_dir, "libdpsr.stamp")
    fp = _fingerprint(extra)
    if not force and os.path.exists(lib) and os.path.exists(stamp):
        with open(stamp) as f:
            if f.read().strip() == fp and os.path.exists(os.path.join(build_dir, BIND_NAME)):
                return lib
    nvcc = _nvcc()
    objs = []

    def compile_one(src):
        obj = os.path.join(build_dir, os.path.splitext(src)[0] + ".o")
        cmd = [nvcc, *ARCH, *FLAGS, *extra, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{res.stderr[-6000:]}")
        if verbose and res.stderr:
            sys.stderr.write(res.stderr)
        return obj

    comp, libs = _bind_flags()
    bind_obj = os.path.join(build_dir, "torch_bind.o")

    def run(cmd, what):
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(f"{what} failed:\n{res.stderr[-6000:]}")

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES) + 1) as ex:
        bind = ex.submit(run, ["g++", *comp, "-c", os.path.join(CSRC, BIND), "-o", bind_obj], f"g++ on {BIND}")
        objs = list(ex.map(compile_one, SOURCES))
        bind.result()
    tmp = lib + f".tmp{os.getpid()}"
    cmd = [nvcc, *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link failed:\n{res.stderr[-4000:]}")
    os.replace(tmp, lib)
    ext = os.path.join(build_dir, BIND_NAME)
    tmp = ext + f".tmp{os.getpid()}"
    run(["g++", "-shared", "-o", tmp, bind_obj, f"-L{build_dir}", *libs], "link of the PyTorch binding")
    os.replace(tmp, ext)
    with open(stamp, "w") as f:
        f.write(fp)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug="--debug" in sys.argv))
