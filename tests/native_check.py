"""Compiles the check programs of tests/ against the library's sources and objects."""
import os
import shutil
import subprocess

from paper_2510_02635_gb300 import build as gbuild

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def nvcc():
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else shutil.which("nvcc")


def _compile(source, directory, objs=()) -> str:
    exe = os.path.join(str(directory), source[:-3])
    cmd = [nvcc(), "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
           "-I", os.path.join(ROOT, "include"), "-I", gbuild.CSRC, os.path.join(HERE, source),
           *objs, "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return exe


def compile_anchored_check(directory) -> str:
    return _compile("anchored_check.cu", directory)


def compile_solve_check(directory) -> str:
    gbuild.build()
    objs = [os.path.join(gbuild.BUILD, f) for f in ("fbsde_kernels_f32.o", "fbsde_kernels_f64.o")]
    if not all(os.path.exists(o) for o in objs):   # a library that came without its objects
        gbuild.build(force=True)
    return _compile("solve_check.cu", directory, objs)
