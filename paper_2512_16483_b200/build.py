"""Builds libfvar.so (the C-ABI library) in-tree with nvcc for sm_100a, and _calls.so (the binding's short calls) beside it."""
from __future__ import annotations

import concurrent.futures
import importlib.metadata
import importlib.util
import os
import re
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libfvar.so")
CALLS = os.path.join(HERE, "_calls.so")
HEADER = os.path.join(HERE, "..", "include", "fvar.h")
OBJDIR = os.path.join(HERE, "_build")
SOURCES = ("gemm.cu", "gemm_pair.cu", "gemm_skinny.cu", "gemm_flex.cu", "attention.cu", "elementwise.cu", "transition.cu", "lls.cu", "fvar_api.cu", "no_alloc.cu", "schedule.cu")
NVCC_FLAGS = os.environ.get("FVAR_NVCC_EXTRA", "").split() + ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--use_fast_math", "-Xptxas", "-v"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _sources():
    return [s for s in SOURCES if os.path.exists(os.path.join(CSRC, s))]


def _older(target: str, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def _lib_stale() -> bool:
    return _older(LIB, [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != "pycalls.cpp"] + [HEADER])


def _built_for() -> str:
    """What _calls.so fits: its symbols are those of one torch and one Python.  The text stands in the file itself."""
    return "fvar call layer for torch %s, Python %s" % (importlib.metadata.version("torch"), sysconfig.get_python_version())


def calls_built_for() -> str:
    """The same text as the _calls.so that is there has it ('' if it has none)."""
    with open(CALLS, "rb") as f:
        found = re.search(rb"fvar call layer for torch [^\0]*", f.read())
    return found.group().decode() if found else ""


def _calls_stale() -> bool:
    return _older(CALLS, [os.path.join(CSRC, "pycalls.cpp"), HEADER]) or calls_built_for() != _built_for()


def _compile(src: str) -> str:
    obj = os.path.join(OBJDIR, src.replace(".cu", ".o"))
    cmd = [_nvcc(), *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
    p = subprocess.run(cmd, capture_output=True, text=True)
    with open(obj + ".log", "w") as f:
        f.write(" ".join(cmd) + "\n" + p.stdout + p.stderr)
    if p.returncode != 0:
        raise RuntimeError("nvcc failed for %s:\n%s" % (src, p.stderr[-4000:]))
    return obj


def _compile_calls() -> str:
    """csrc/pycalls.cpp: host code against torch's headers, linked to the library beside it."""
    torch_dir = importlib.util.find_spec("torch").submodule_search_locations[0]
    inc, libs = os.path.join(torch_dir, "include"), os.path.join(torch_dir, "lib")
    cuda = os.path.dirname(os.path.dirname(_nvcc())) or "/usr/local/cuda"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", '-DFVAR_BUILT_FOR="%s"' % _built_for(), "-I" + inc, "-I" + os.path.join(inc, "torch", "csrc", "api", "include"),
           "-I" + os.path.join(cuda, "include"), "-I" + sysconfig.get_paths()["include"], os.path.join(CSRC, "pycalls.cpp"), "-o", CALLS,
           "-L" + HERE, "-l:libfvar.so", "-L" + libs, "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python", "-Wl,-rpath,$ORIGIN"]
    p = subprocess.run(cmd, capture_output=True, text=True)
    if p.returncode != 0:
        raise RuntimeError("g++ failed for pycalls.cpp:\n" + p.stderr[-4000:])
    return CALLS


def _build_lib() -> list:
    os.makedirs(OBJDIR, exist_ok=True)
    with concurrent.futures.ThreadPoolExecutor(max_workers=4) as ex:
        objs = list(ex.map(_compile, _sources()))
    cmd = [_nvcc(), "-shared", "-o", LIB, *objs, "-gencode", "arch=compute_100a,code=sm_100a"]
    p = subprocess.run(cmd, capture_output=True, text=True)
    if p.returncode != 0:
        raise RuntimeError("link failed:\n" + p.stderr[-4000:])
    return objs


def build(force: bool = False, verbose: bool = False) -> str:
    objs = _build_lib() if force or _lib_stale() else []
    if force or _calls_stale():
        _compile_calls()
    if verbose:
        for o in objs:
            sys.stdout.write(open(o + ".log").read())
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
