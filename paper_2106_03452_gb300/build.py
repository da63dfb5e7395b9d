"""Build libdpsr.so in-tree with nvcc for sm_103a (GB300), and the PyTorch
binding of its hot calls with g++.

Each .cu translation unit is compiled in parallel, then linked into
paper_2106_03452_gb300/_build/libdpsr.so (nvcc alone: no torch, no cmake);
csrc/torch_bind.cpp becomes _build/_dpsr_torch.so next to it, against the
headers of the installed PyTorch. Without PyTorch, or where that fails, the
library is there all the same, and the Python classes do without the binding.
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
    """PyTorch, or None where there is none."""
    try:
        import torch
    except ImportError:
        return None
    return torch


def _bind_flags(torch):
    """(compile, link) flags of the binding: PyTorch's headers and libraries."""
    root = os.path.dirname(torch.__file__)
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include"),
           INCLUDE]
    abi = f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}"
    comp = ["-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden", abi, *(f"-I{d}" for d in inc)]
    link = [f"-L{os.path.join(root, 'lib')}", "-lc10", "-lc10_cuda", "-ltorch", "-ltorch_cpu", "-ltorch_cuda",
            "-ltorch_python", "-ldpsr", "-Wl,-rpath,$ORIGIN"]
    return comp, link


def _fingerprint(files, flags) -> str:
    h = hashlib.sha256()
    for p in files:
        h.update(os.path.basename(p).encode())
        with open(p, "rb") as f:
            h.update(f.read())
    h.update(" ".join(flags).encode())
    return h.hexdigest()


def _files(d):
    return [p for n in sorted(os.listdir(d)) if os.path.isfile(p := os.path.join(d, n))]


def _stamped(path, stamp, fp) -> bool:
    if not (os.path.exists(path) and os.path.exists(stamp)):
        return False
    with open(stamp) as f:
        return f.read().strip() == fp


def _write(stamp, fp):
    with open(stamp, "w") as f:
        f.write(fp)


def _run(cmd, what, verbose=False):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"{what} failed:\n{res.stderr[-6000:]}")
    if verbose and res.stderr:
        sys.stderr.write(res.stderr)


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    """Compile libdpsr.so; with debug=True the bounds-checking variant
    (-DDPSR_DEBUG_CHECKS) into its own folder. Then the PyTorch binding."""
    build_dir, lib = (BUILD_DEBUG, LIB_DEBUG) if debug else (BUILD, LIB)
    extra = ["-DDPSR_DEBUG_CHECKS=1"] if debug else []
    os.makedirs(build_dir, exist_ok=True)
    torch, ext = _torch(), os.path.join(build_dir, BIND_NAME)
    stamp, bind_stamp = os.path.join(build_dir, "libdpsr.stamp"), ext + ".stamp"
    source, bind_obj = os.path.join(CSRC, BIND), os.path.join(build_dir, "torch_bind.o")
    fp = _fingerprint([p for p in _files(CSRC) + _files(INCLUDE) if p != source], ARCH + FLAGS + extra)
    make_lib = force or not _stamped(lib, stamp, fp)
    make_bind = False
    if torch is not None:
        comp, link = _bind_flags(torch)
        # the version in plain text, first: libdpsr.binding() compares it
        bind_fp = f"{torch.__version__}\n{_fingerprint([source, *_files(INCLUDE)], comp + link)}"
        make_bind = force or not _stamped(ext, bind_stamp, bind_fp)

    def compile_one(src):
        obj = os.path.join(build_dir, os.path.splitext(src)[0] + ".o")
        _run([_nvcc(), *ARCH, *FLAGS, *extra, *(["-Xptxas=-v"] if verbose else []), "-c", os.path.join(CSRC, src),
              "-o", obj], f"nvcc on {src}", verbose)
        return obj

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES) + 1) as ex:
        bind = ex.submit(_run, ["g++", *comp, "-c", source, "-o", bind_obj], f"g++ on {BIND}") if make_bind else None
        if make_lib:
            objs = list(ex.map(compile_one, SOURCES))
            tmp = lib + f".tmp{os.getpid()}"
            _run([_nvcc(), *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"], "link")
            os.replace(tmp, lib)
            _write(stamp, fp)
    if make_bind:
        try:
            bind.result()
            tmp = ext + f".tmp{os.getpid()}"
            _run(["g++", "-shared", "-o", tmp, bind_obj, f"-L{build_dir}", *link], "link of the PyTorch binding")
            os.replace(tmp, ext)
            _write(bind_stamp, bind_fp)
        except (RuntimeError, OSError) as e:
            if os.path.exists(ext):
                os.remove(ext)  # one of other sources, or of another PyTorch
            sys.stderr.write(f"libdpsr is built without its PyTorch binding: {e}\n")
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug="--debug" in sys.argv))
