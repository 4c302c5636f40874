"""Builds libgformer.so in-tree with nvcc for sm_100a, and _fastcall.so beside it with g++ (no JIT cache).

Usage: python -m paper_2412_19829_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB = os.path.join(HERE, "libgformer.so")
FASTCALL = os.path.join(HERE, "_fastcall.so")  # the binding's calls as a module (csrc/fastcall.cpp)
SOURCES = ["api.cu", "simt_kernels.cu", "simt_tiled.cu", "tma_host.cu", "host_state.cu", "tc_window.cu", "tc_linear.cu", "tc_linear_self.cu", "noalloc.cu", "partition.cu", "tc_favor.cu"]
ARCH = ["-gencode", "arch=compute_100a,code=sm_100a"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; libgformer cannot be built")


def _sources():
    return [os.path.join(CSRC, s) for s in SOURCES if os.path.exists(os.path.join(CSRC, s))]


def _older(target: str, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(p) > os.path.getmtime(target) for p in deps)


def _stale() -> bool:
    headers = [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    return (_older(LIB, _sources() + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))] + headers)
            or _older(FASTCALL, [os.path.join(CSRC, "fastcall.cpp")] + headers) or _fastcall_built_for() != fastcall_target())


def fastcall_target() -> str:
    """What the module is built against, which it is no good without."""
    import torch

    return f"{sys.implementation.cache_tag}, torch {torch.__version__}"


def _fastcall_built_for() -> str:
    try:
        with open(os.path.join(HERE, "build", "_fastcall.target")) as f:
            return f.read()
    except OSError:
        return ""


def _build_fastcall(out: str) -> subprocess.Popen:
    import sysconfig

    import torch

    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    inc = [INCLUDE, sysconfig.get_paths()["include"], os.path.join(root, "include"),
           os.path.join(root, "include", "torch", "csrc", "api", "include"), os.path.join(cuda, "include")]
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
           f'-DGF_BUILT_FOR="{fastcall_target()}"']
    cmd += [x for i in inc for x in ("-I", i)] + [os.path.join(CSRC, "fastcall.cpp"), "-o", out]
    cmd += ["-L", os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-ldl"]
    return subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    nvcc = _nvcc()
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    flags = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC] + ARCH
    if verbose:
        flags += ["-Xptxas", "-v"]
    objs = [os.path.join(objdir, os.path.basename(src)[:-3] + ".o") for src in _sources()]
    # (linked beside the objects, which git ignores, and moved into place when complete)
    lib_tmp, fast_tmp = (os.path.join(objdir, f"{os.path.basename(x)}.{os.getpid()}.tmp") for x in (LIB, FASTCALL))
    try:
        procs = [(src, subprocess.Popen([nvcc, "-c", src, "-o", obj] + flags,
                                        stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True))
                 for src, obj in zip(_sources(), objs)]
        # The library needs neither torch nor g++, and binding.py does without the module.
        try:
            fast = _build_fastcall(fast_tmp)
        except (ImportError, OSError) as e:
            fast = None
            print(f"_fastcall.so not built: {e}", file=sys.stderr)
        failed = False
        for src, p in procs + ([("fastcall.cpp", fast)] if fast else []):
            out, _ = p.communicate()
            if out.strip() and (verbose or p.returncode != 0):
                print(out, file=sys.stderr)
            failed |= p.returncode != 0 and p is not fast
        if failed:
            raise RuntimeError("nvcc failed")
        subprocess.check_call([nvcc, "-shared", "-o", lib_tmp] + objs + ARCH + ["-cudart", "static"])
        os.replace(lib_tmp, LIB)
        if fast is not None and fast.returncode == 0:
            os.replace(fast_tmp, FASTCALL)
            with open(os.path.join(objdir, "_fastcall.target"), "w") as f:
                f.write(fastcall_target())
        elif os.path.exists(FASTCALL):  # (made for another library)
            os.remove(FASTCALL)
    finally:
        for x in (lib_tmp, fast_tmp):
            if os.path.exists(x):
                os.remove(x)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
