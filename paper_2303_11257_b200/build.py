"""Builds libunitscale.so (sm_100a) and its Python binding in-tree with nvcc.

    python -m paper_2303_11257_b200.build [--force]
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libunitscale.so")
BINDING = os.path.join(HERE, "_binding.so")
SOURCES = ["host.cu", "elementwise.cu", "softmax.cu", "layernorm.cu", "diagnostics.cu", "gemm.cu", "gemm_group.cu", "gemm_split.cu", "ffn_hidden.cu", "static_ws.cu", "attention.cu", "attention_grads.cu"]
# (operand bytes, A MN-major, B MN-major): forward, backward-input, backward-weight for FP8 and 16-bit operands
GEMM_PARTS = [(1, 0, 1), (1, 0, 0), (1, 1, 1), (2, 0, 1), (2, 0, 0), (2, 1, 1)]
HEADERS = ["common.cuh", "rowwise.cuh", "sm100.cuh", "gemm_kernel.cuh", "gemm_group.cuh", "gemm_split.cuh", "gemm_launch.h", "attention_host.h", "gemm_inst.cu", "host.h", os.path.join("..", "..", "include", "unitscale.h")]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def built_for() -> str:
    """The Python and torch whose headers and libraries the binding is built with; it holds this text (built_for in binding.cpp)."""
    import torch
    return f"us-binding-for python {sys.version_info[0]}.{sys.version_info[1]} torch {torch.__version__};"


def _stale() -> bool:
    if not (os.path.exists(LIB) and os.path.exists(BINDING)):
        return True
    with open(BINDING, "rb") as f:                              # it cannot be imported to be asked: another torch may lack its symbols
        if built_for().encode() not in f.read():
            return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(BINDING))
    deps = [os.path.join(CSRC, f) for f in SOURCES + HEADERS + ["binding.cpp"]] + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def _compile(args):
    res = subprocess.run(args, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + " ".join(args) + "\n" + res.stdout + res.stderr)
    return res.stderr


def _binding_jobs(obj):
    """Compiles and links the Python module (argument marshalling; torch's headers, and symbols of the torch that imports it)."""
    import sysconfig
    import torch
    top = os.path.dirname(os.path.abspath(torch.__file__))
    compile_ = [_nvcc(), "-std=c++17", "-O2", "-x", "c++", f'-DUS_BUILT_FOR="{built_for()}"', "-Xcompiler", f"-fPIC,-fvisibility=hidden,-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
                "-I", sysconfig.get_paths()["include"], "-I", os.path.join(top, "include"), "-c", "-o", obj, os.path.join(CSRC, "binding.cpp")]
    link = [_nvcc(), "-shared", "-o", BINDING, obj, LIB, "-L", os.path.join(top, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lcudart",
            "-Xlinker", "-rpath,$ORIGIN"]
    return compile_, link


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile the library and the binding if one is missing, older than its sources or built for another Python or torch; returns
    the library's path.

    Every translation unit is compiled to an object in parallel (gemm_inst.cu once per operand
    width and layout), then linked into libunitscale.so next to this file."""
    if not force and not _stale():
        return LIB
    from concurrent.futures import ThreadPoolExecutor
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    common = [_nvcc(), "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
              "-Xcompiler", "-fPIC", "-Xptxas", "-v" if verbose else "-O3", "-c"]
    jobs, objs = [], []
    for f in SOURCES:
        o = os.path.join(objdir, f.replace(".cu", ".o"))
        objs.append(o)
        jobs.append(common + ["-o", o, os.path.join(CSRC, f)])
    for es, amn, bmn in GEMM_PARTS:
        o = os.path.join(objdir, f"gemm_inst_{es}_{amn}_{bmn}.o")
        objs.append(o)
        jobs.append(common + [f"-DUS_INST_ES={es}", f"-DUS_INST_AMN={amn}", f"-DUS_INST_BMN={bmn}", "-o", o,
                              os.path.join(CSRC, "gemm_inst.cu")])
    compile_binding, link_binding = _binding_jobs(os.path.join(objdir, "binding.o"))
    with ThreadPoolExecutor(max_workers=min(len(jobs), os.cpu_count() or 4)) as pool:
        logs = list(pool.map(_compile, [compile_binding] + jobs))
    _compile([_nvcc(), "-shared", "-o", LIB, "-Xlinker", "-soname,libunitscale.so"] + objs + ["-lcudart"])
    _compile(link_binding)
    if verbose:
        print("\n".join(logs))
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
