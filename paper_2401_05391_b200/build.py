"""Build the segkv C-ABI shared library in-tree with nvcc for sm_100a."""
from __future__ import annotations

import glob
import os
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libsegkv.so")
# the same library with per-CTA time stamps compiled in (read by paper_2401_05391_b200/timeline.py);
# never loaded by the binding, the tests or the benchmark
LIB_TIMELINE = os.path.join(PKG, "libsegkv_timeline.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--use_fast_math",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
] + os.environ.get("SEGKV_NVCC_FLAGS", "").split()


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(p) > t for p in deps)


def hot_path() -> str:
    """Where the binding's extension module (csrc/segkv_hot.cpp) belongs for the torch and the Python that run here: it reads
    torch's C++ objects, so each version of either has a file of its own and never loads another's."""
    import sysconfig

    import torch
    return os.path.join(PKG, f"segkv_hot.torch-{torch.__version__}{sysconfig.get_config_var('EXT_SUFFIX')}")


def build_hot(force: bool = False) -> str:
    """Compile csrc/segkv_hot.cpp into the extension module at hot_path() (no-op when up to date)."""
    import sysconfig

    import torch
    src, out = os.path.join(CSRC, "segkv_hot.cpp"), hot_path()
    if not force and os.path.exists(out) and os.path.getmtime(out) >= os.path.getmtime(src):
        return out
    root = os.path.dirname(torch.__file__)
    tmp = out + f".{os.getpid()}.tmp"
    subprocess.check_call([
        os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
        f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
        "-I", os.path.join(root, "include"), "-I", sysconfig.get_paths()["include"],
        "-I", os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include"), src, "-o", tmp,
        "-L", os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"])
    os.replace(tmp, out)
    return out


def build(force: bool = False, verbose: bool = False, timeline: bool = False) -> str:
    """Compile every .cu under csrc/ into libsegkv.so (no-op when up to date), then the binding's extension module where torch and a
    C++ compiler allow it (the library needs neither, and the binding runs without it).  `timeline` builds the
    instrumented copy libsegkv_timeline.so instead."""
    if timeline:
        return _build_lib(LIB_TIMELINE, force, verbose, timeline)
    lib = _build_lib(LIB, force, verbose)
    try:
        build_hot(force)
    except (ImportError, OSError, subprocess.CalledProcessError) as e:
        sys.stderr.write(f"the decode loop's extension module was not built ({e}): its calls go through ctypes\n")
    return lib


def _build_lib(lib: str, force: bool, verbose: bool, timeline: bool = False) -> str:
    if not (force or _stale(lib)):
        return lib
    objs = []
    procs = []
    for src in sources():
        obj = os.path.splitext(src)[0] + (".tl.o" if timeline else ".o")
        cmd = [NVCC, *FLAGS, *(["-DSEGKV_TIMELINE"] if timeline else []), "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(f"--- {os.path.basename(src)}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = lib + f".{os.getpid()}.tmp"
    subprocess.check_call([NVCC, "-shared", "-gencode", "arch=compute_100a,code=sm_100a",
                           "-cudart", "static", "-o", tmp, *objs])
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, timeline="--timeline" in sys.argv))
