"""In-tree build of the CUDA library (sm_100a only) and of its torch binding: ``python -m paper_2609_24433_b200.build``."""
from __future__ import annotations

import importlib.metadata
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libfq_b200.so")
SOURCES = ["fq_api.cu", "act_quant.cu", "act_quant_ring.cu", "gemm_simt.cu", "gemm_tcgen05.cu", "linear_fused.cu", "fq_static.cu", "linear_wonly.cu", "composite.cu", "gptq.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]
BINDING = os.path.join(HERE, "_fq_torch" + sysconfig.get_config_var("EXT_SUFFIX"))
BINDING_TORCH = os.path.join(HERE, "_fq_torch.built")     # the torch that the binding was compiled against


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build_binding(force: bool = False) -> str:
    """The CPython module over the library: plain C++ against torch's headers, linked to the library next to it."""
    src = os.path.join(CSRC, "torch_binding.cpp")
    version = importlib.metadata.version("torch")         # (its headers are part of the source: another torch, another module)
    built = open(BINDING_TORCH).read().strip() if os.path.exists(BINDING_TORCH) else ""
    if force or built != version or _stale(BINDING, [src, os.path.join(ROOT, "include", "fq.h")]):
        import torch
        t = os.path.dirname(torch.__file__)
        inc = [os.path.join(ROOT, "include"), os.path.join(t, "include"), os.path.join(t, "include", "torch", "csrc", "api", "include"),
               sysconfig.get_paths()["include"], "/usr/local/cuda/include"]
        subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared"] + [f for d in inc for f in ("-I", d)] +
                       [src, "-o", BINDING, "-L", HERE, "-l:" + os.path.basename(LIB), "-L", os.path.join(t, "lib"), "-lc10",
                        "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python", "-Wl,-rpath,$ORIGIN"], check=True)
        with open(BINDING_TORCH, "w") as f:
            f.write(version + "\n")
    return BINDING


def build(force: bool = False, verbose: bool = False) -> str:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(ROOT, "include", "fq.h"))
    objs = []
    relink = force
    jobs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(CSRC, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + headers):
            jobs.append([nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", s, "-o", o])
            relink = True
    if jobs:      # the translation units are independent: compile them side by side
        from concurrent.futures import ThreadPoolExecutor
        with ThreadPoolExecutor(max_workers=min(len(jobs), os.cpu_count() or 1)) as pool:
            for done in pool.map(lambda cmd: subprocess.run(cmd, check=True), jobs):
                pass
    if relink or _stale(LIB, objs):
        subprocess.run([nvcc, "-shared", "-o", LIB] + objs, check=True)
    build_binding(force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
