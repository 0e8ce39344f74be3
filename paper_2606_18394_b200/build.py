"""Builds libjet.so (the C-ABI library, nvcc for sm_100a) and the binding's CPython extension in-tree."""
from __future__ import annotations

import json
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libjet.so")
# the binding's argument marshalling (a CPython extension linked against libjet.so and torch)
EXT = os.path.join(PKG, "_jetcall" + sysconfig.get_config_var("EXT_SUFFIX"))
# what the extension was built for: it links torch's libraries, whose C++ interface changes between versions
STAMP = os.path.join(PKG, "build", "jetcall.json")
SOURCES = ["jet_api.cu", "tree_build.cu", "tree_verify_attn.cu", "tree_accept.cu", "tree_accept_sample.cu",
           "kv_compact.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden"]
# Only the attention kernel is built with fast math (approximate exp2 / division, subnormals flushed): its
# outputs carry a tolerance.  The tree, acceptance and commit kernels promise bit-exact results on IEEE
# fp32 adds and compares -- subnormal log-probabilities and logits included -- and are built without it.
FAST_MATH_SOURCES = {"tree_verify_attn.cu"}


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _environment() -> dict:
    import torch
    return {"torch": str(torch.__version__), "cxx11_abi": int(torch._C._GLIBCXX_USE_CXX11_ABI), "python": sys.version.split()[0]}


def needs_build() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(EXT):
        return True
    try:
        with open(STAMP) as f:
            if json.load(f) != _environment():
                return True
    except (OSError, ValueError):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(EXT))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "jet.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _extension_commands(obj: str) -> tuple[list[str], list[str]]:
    """Compile and link command of the CPython extension."""
    import torch
    troot = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    inc = [os.path.join(ROOT, "include"), sysconfig.get_paths()["include"], os.path.join(troot, "include"),
           os.path.join(troot, "include", "torch", "csrc", "api", "include"), os.path.join(cuda, "include")]
    compile_cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden",
                   f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                   f'-DJET_TORCH_VERSION="{torch.__version__}"', *(x for i in inc for x in ("-I", i)),
                   "-c", os.path.join(CSRC, "jetcall.cpp"), "-o", obj]
    link_cmd = ["g++", "-shared", "-o", EXT, obj, "-L", PKG, "-l:libjet.so", "-L", os.path.join(troot, "lib"),
                "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-Wl,-rpath,$ORIGIN"]
    return compile_cmd, link_cmd


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile everything under csrc/ into objects, link libjet.so and the CPython extension.  Returns libjet.so's path."""
    if not force and not needs_build():
        return LIB
    objdir = os.path.join(PKG, "build")
    os.makedirs(objdir, exist_ok=True)
    procs = []
    objs = []
    for src in SOURCES:
        obj = os.path.join(objdir, src.replace(".cu", ".o"))
        objs.append(obj)
        cmd = [_nvcc(), *NVCC_FLAGS, *(["--use_fast_math"] if src in FAST_MATH_SOURCES else []),
               "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    ext_obj = os.path.join(objdir, "jetcall.o")
    ext_compile, ext_link = _extension_commands(ext_obj)
    procs.append(("jetcall.cpp", subprocess.Popen(ext_compile, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(f"--- {src}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("compiling libjet.so or its Python binding failed")
    link = [_nvcc(), "-shared", "-o", LIB, *objs, "-gencode", "arch=compute_100a,code=sm_100a",
            "-Xcompiler", "-fPIC"]
    subprocess.run(link, check=True)
    subprocess.run(ext_link, check=True)
    with open(STAMP, "w") as f:
        json.dump(_environment(), f)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
