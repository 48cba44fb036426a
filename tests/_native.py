"""Small CUDA programs against the library's headers, for what no public call shows."""
import os
import subprocess

from paper_1411_4510_gb300 import build as B


def compile_program(source: str, folder) -> str:
    """Compiles a program for sm_103a (host code runs without a GPU) and returns its path."""
    src, exe = os.path.join(str(folder), "prog.cu"), os.path.join(str(folder), "prog")
    with open(src, "w") as fh:
        fh.write(source)
    cmd = [B._nvcc(), *B.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-I" + B.INCLUDE, "-I" + B.CSRC,
           "-o", exe, src]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return exe


def run_program(exe: str, *args, timeout=120) -> str:
    r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=timeout)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
