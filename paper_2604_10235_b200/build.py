"""Builds libcodecomp.so (sm_100a) and the extension that calls it from Python, in-tree, with nvcc."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB_DIR = os.path.join(HERE, "lib")
LIB_PATH = os.path.join(LIB_DIR, "libcodecomp.so")
# Python extension that marshals the calls; the suffix names the interpreter it is built for
CALL_PATH = os.path.join(LIB_DIR, "_cccall" + sysconfig.get_config_var("EXT_SUFFIX"))
SOURCES = ["api.cu", "score_simt.cu", "score_tc.cu", "fuse_pool.cu", "select.cu", "select_cluster.cu", "compact.cu",
           "str_score.cu", "planner.cu", "ppl.cu", "exp_probe.cu"]


def nvcc_path() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; libcodecomp.so cannot be built")


def _stale() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(CALL_PATH):
        return True
    built = min(os.path.getmtime(LIB_PATH), os.path.getmtime(CALL_PATH))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps.append(os.path.join(ROOT, "include", "codecomp.h"))
    return any(os.path.getmtime(d) > built for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles every CUDA source for sm_100a and links the shared library."""
    if not force and not _stale():
        return LIB_PATH
    os.makedirs(LIB_DIR, exist_ok=True)
    obj_dir = os.path.join(HERE, "_build")
    os.makedirs(obj_dir, exist_ok=True)
    nvcc = nvcc_path()
    common = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3",
              "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
              "-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if verbose:
        common += ["-Xptxas", "-v"]
    call = [nvcc, "-shared", "-cudart", "none", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
            "-I", sysconfig.get_paths()["include"], "-I", os.path.join(ROOT, "include"), os.path.join(CSRC, "py_call.cpp"), "-o", CALL_PATH]
    procs = [("py_call.cpp", subprocess.Popen(call, stdout=subprocess.PIPE, stderr=subprocess.STDOUT,
                                              text=True))]
    objs = []
    for src in SOURCES:
        obj = os.path.join(obj_dir, src.replace(".cu", ".o"))
        objs.append(obj)
        procs.append((src, subprocess.Popen(common + ["-c", os.path.join(CSRC, src), "-o", obj],
                                            stdout=subprocess.PIPE, stderr=subprocess.STDOUT,
                                            text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(f"--- {src}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed; see the compiler output above")
    link = [nvcc, "-shared", "-o", LIB_PATH] + objs + ["-cudart", "static"]
    res = subprocess.run(link, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if res.returncode != 0:
        raise RuntimeError("link failed:\n" + res.stdout)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
