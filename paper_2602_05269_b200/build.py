"""Build libhgf_b200.so (sm_100a, nvcc) and the binding's native part (_hgf_python, g++) in-tree.  Run as `python -m paper_2602_05269_b200.build`."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libhgf_b200.so")
OBJ_DIR = os.path.join(HERE, "_build")
SOURCES = ["hgf_api.cu", "hgf_pack.cu", "hgf_prologue.cu", "hgf_decode.cu", "hgf_decode_small.cu", "hgf_decode_tc.cu", "hgf_prefill.cu", "hgf_attention.cu", "hgf_backward.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def module_path() -> str:
    """The binding's native part: one for each Python and torch, whose binary interfaces it is compiled against."""
    import torch
    return os.path.join(HERE, f"_hgf_python.{sysconfig.get_config_var('SOABI')}.torch-{torch.__version__}.so")


def _deps(src: str):
    return [src, os.path.join(CSRC, "hgf_common.cuh"), os.path.join(CSRC, "hgf_tc.cuh"), os.path.join(CSRC, "hgf_warp.cuh"), os.path.join(HERE, "..", "include", "hgf.h")]


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source for sm_100a and link the shared library.  Returns its path."""
    os.makedirs(OBJ_DIR, exist_ok=True)
    nvcc = _nvcc()
    flags = list(NVCC_FLAGS)
    if verbose:
        flags += ["-Xptxas", "-v"]
    srcs = [s for s in SOURCES if os.path.exists(os.path.join(CSRC, s))]
    jobs = []
    for s in srcs:
        src = os.path.join(CSRC, s)
        obj = os.path.join(OBJ_DIR, s.replace(".cu", ".o"))
        newest = max(os.path.getmtime(d) for d in _deps(src))
        if force or verbose or not os.path.exists(obj) or os.path.getmtime(obj) < newest:
            jobs.append([nvcc, *flags, "-c", src, "-o", obj])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode:
            sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        if r.returncode:
            raise RuntimeError(f"{os.path.basename(cmd[0])} failed: " + " ".join(cmd))

    with ThreadPoolExecutor(max_workers=4) as ex:
        list(ex.map(run, jobs))
    objs = [os.path.join(OBJ_DIR, s.replace(".cu", ".o")) for s in srcs]
    if jobs or force or not os.path.exists(LIB):
        tmp = LIB + f".tmp{os.getpid()}"
        run([nvcc, "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a"])
        os.replace(tmp, LIB)

    src = os.path.join(CSRC, "hgf_python.cpp")
    newest = max(os.path.getmtime(d) for d in (src, os.path.join(HERE, "..", "include", "hgf.h")))
    module = module_path()
    if force or not os.path.exists(module) or os.path.getmtime(module) < newest:
        import torch
        t = os.path.dirname(torch.__file__)
        cuda = os.path.join(os.path.dirname(os.path.dirname(nvcc)) if os.path.isabs(nvcc) else "/usr/local/cuda", "include")
        tmp = module + f".tmp{os.getpid()}"
        run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-I{t}/include", f"-I{t}/include/torch/csrc/api/include", f"-I{cuda}",
             f"-I{sysconfig.get_paths()['include']}", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}", src, "-o", tmp,
             f"-L{t}/lib", "-ltorch_python", "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda"])
        os.replace(tmp, module)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
