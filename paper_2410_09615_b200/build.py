"""In-tree build of libslim.so (nvcc, sm_100a only) and of the Python call path on it (g++, torch's headers)."""
from __future__ import annotations

import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libslim.so")
NATIVE = os.path.join(HERE, "_slim_native.so")
SOURCES = ["api.cu", "pack.cu", "repack.cu", "fwd_simple.cu", "fwd_small.cu", "fwd_prefill.cu",
           "fwd_noalloc.cu", "adapter_q.cu", "quant_search.cu", "mask.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
              "-Xcompiler", "-fPIC", "--use_fast_math"]


def _older(target: str, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def _stale() -> bool:
    return _older(LIB, [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")] + [os.path.join(INCLUDE, "slim.h")])


def _cudart(torch_root: str):
    """The CUDA runtime that torch itself has loaded, by its file name (the module shares its context and streams)."""
    import glob
    near = glob.glob(os.path.join(os.path.dirname(torch_root), "nvidia", "cuda_runtime", "lib", "libcudart.so*"))
    lib = near[0] if near else "/usr/local/cuda/lib64/libcudart.so"
    return ["-L" + os.path.dirname(lib), "-l:" + os.path.basename(lib)]


def build_native(force: bool = False) -> str:
    """Compile ``csrc/native.cpp`` into ``_slim_native.so`` (for the interpreter and the torch that run this)."""
    src = os.path.join(CSRC, "native.cpp")
    if not force and not _older(NATIVE, [src]):
        return NATIVE
    import sysconfig
    import torch
    root = os.path.dirname(torch.__file__)
    dirs = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
            os.environ.get("CUDA_HOME", "/usr/local/cuda") + "/include", sysconfig.get_paths()["include"]]
    tmp = NATIVE + f".tmp{os.getpid()}"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                           *[f"-I{d}" for d in dirs], src, "-o", tmp, "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch",
                           "-ltorch_cpu", "-ltorch_cuda", "-lc10", "-lc10_cuda", *_cudart(root)])
    os.replace(tmp, NATIVE)
    return NATIVE


def build(force: bool = False, verbose: bool = False, defines=(), out: str | None = None) -> str:
    """Compile every CUDA source into ``libslim.so`` next to this file.

    ``defines``: extra ``-D`` macros, the kernels' optional hooks: ``SLIM_PREFILL_TRACE`` (per-CTA timeline
    of the prefill kernel, read back with the ``slim_debug_read_ptrace`` function such a build exports).  A
    build with hooks goes to ``out`` (required then), never to the library the package loads by default."""
    if defines and not out:
        raise ValueError("a build with extra defines needs its own output path")
    if not defines:
        build_native(force)
    if not defines and not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    bdir = os.path.join(HERE, "_build" + ("_" + "_".join(sorted(defines)) if defines else ""))
    os.makedirs(bdir, exist_ok=True)
    procs = []
    for src in SOURCES:
        obj = os.path.join(bdir, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, *[f"-D{d}" for d in defines], "-I", INCLUDE, "-I", CSRC, "-c", os.path.join(CSRC, src),
               "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    for src, pr in procs:
        log, _ = pr.communicate()
        if pr.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{log}")
        if verbose and log:
            print(log)
    target = out or LIB
    tmp = target + f".tmp{os.getpid()}"
    subprocess.check_call([nvcc, "-shared", "-o", tmp, *objs, "-cudart", "static"])
    os.replace(tmp, target)
    return target


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
