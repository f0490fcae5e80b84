"""Builds ``libdsla.so`` in-tree with nvcc for sm_100a (cross-compiles without a GPU), and beside it the extension
module ``_native`` (argument marshalling for torch tensors, plain C++)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdsla.so")
NATIVE = os.path.join(HERE, "_native.so")
SOURCES = ["dsla_api.cu", "dsla_decode.cu", "dsla_gate_project.cu", "dsla_prefill_simt.cu", "dsla_prefill_recurrent.cu", "dsla_prefill_summary.cu", "dsla_prefill_tc.cu",
           "dsla_prefill_tc_pair.cu", "dsla_prefill_vec.cu", "dsla_static_ws.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
              "-I", CSRC]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(NATIVE):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(NATIVE))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "dsla.h"), __file__]
    return any(os.path.getmtime(d) > t for d in deps)


def _native_cmds(obj: str, out: str):
    """Compile and link commands of the extension module (links against libdsla.so next to it and torch's libraries)."""
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    inc = [os.path.join(ROOT, "include"), os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    compile_ = ["g++", "-O2", "-std=c++17", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                *[x for i in inc for x in ("-I", i)], "-c", os.path.join(CSRC, "dsla_py.cpp"), "-o", obj]
    link = ["g++", "-shared", "-o", out, obj, "-L", HERE, "-ldsla", "-L", os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu",
            "-lc10", "-lc10_cuda", "-Wl,-rpath,$ORIGIN"]
    return compile_, link


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    procs = []
    objs = []
    for src in SOURCES:
        obj = os.path.join(objdir, src.replace(".cu", ".o"))
        objs.append(obj)
        cmd = [_nvcc(), *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    native_obj, native_tmp = os.path.join(objdir, "dsla_py.o"), NATIVE + f".{os.getpid()}.tmp"
    native_compile, native_link = _native_cmds(native_obj, native_tmp)
    procs.append(("dsla_py.cpp", subprocess.Popen(native_compile, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(f"--- nvcc {src}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("compiling libdsla.so failed")
    tmp = LIB + f".{os.getpid()}.tmp"
    subprocess.check_call([_nvcc(), "-shared", "-o", tmp, *objs, "-cudart", "static"])
    os.replace(tmp, LIB)
    subprocess.check_call(native_link)
    os.replace(native_tmp, NATIVE)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
