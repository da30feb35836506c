"""In-tree build of libmemdecay.so for sm_103a (nvcc; no cmake).

The translation units compile in parallel, then link into one shared library
next to this file; the Python module of the per-step calls (_calls, plain C,
named for the interpreter) lands beside it, unless Python's headers are missing:
those calls then go through ctypes.  Run as a module or call build()."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB_PATH = os.path.join(HERE, "libmemdecay.so")
BINDING_PATH = os.path.join(HERE, "_calls" + sysconfig.get_config_var("EXT_SUFFIX"))
OBJ_DIR = os.path.join(HERE, "_build")
SOURCES = ["md_host.cpp", "md_attn.cu", "md_attn_cluster.cu", "md_state.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
         "--expt-relaxed-constexpr", "-I", INCLUDE]


def _deps():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files.append(os.path.join(INCLUDE, "memdecay.h"))
    files.append(os.path.abspath(__file__))
    return files


def python_include():
    """The folder of Python.h, or None."""
    path = sysconfig.get_paths()["include"]
    return path if os.path.exists(os.path.join(path, "Python.h")) else None


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False) -> str:
    newest = max(os.path.getmtime(p) for p in _deps())
    include = python_include()
    made = (LIB_PATH, BINDING_PATH) if include else (LIB_PATH,)
    if not force and all(os.path.exists(p) and os.path.getmtime(p) >= newest for p in made):
        return LIB_PATH
    os.makedirs(OBJ_DIR, exist_ok=True)

    def compile_one(src):
        obj = os.path.join(OBJ_DIR, src + ".o")
        cmd = ["nvcc", *ARCH, *FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if ptxas_info and src.endswith(".cu"):
            cmd.insert(1, "-Xptxas=-v")
        if verbose:
            print(" ".join(cmd), flush=True)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0 or (ptxas_info and r.stderr):
            sys.stderr.write(r.stderr)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
        return obj

    def compile_binding():
        if not include:
            return
        cmd = ["gcc", "-O2", "-Wall", "-shared", "-fPIC", "-I", include, "-I", INCLUDE,
               os.path.join(CSRC, "md_binding.c"), "-o", BINDING_PATH + ".tmp", "-ldl"]
        if verbose:
            print(" ".join(cmd), flush=True)
        subprocess.run(cmd, check=True)
        os.replace(BINDING_PATH + ".tmp", BINDING_PATH)

    with ThreadPoolExecutor(max_workers=len(SOURCES) + 1) as ex:
        binding = ex.submit(compile_binding)
        objs = list(ex.map(compile_one, SOURCES))
        binding.result()
    tmp = LIB_PATH + ".tmp"
    cmd = ["nvcc", *ARCH, "-shared", "-o", tmp, *objs, "-cudart", "static"]
    if verbose:
        print(" ".join(cmd), flush=True)
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv)
    print(LIB_PATH)
