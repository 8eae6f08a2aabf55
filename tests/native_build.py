"""Host programs of the tests that call the library's host code directly (no GPU needed)."""
import os
import subprocess

from paper_1004_0023_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def compile_host(name, out_dir):
    """tests/native/<name>.cu linked against libpt.so; returns the program's path."""
    build.build()
    exe = os.path.join(str(out_dir), name)
    lib_dir = os.path.dirname(build.LIB)
    cmd = [build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, "-o", exe,
           os.path.join(ROOT, "tests", "native", name + ".cu"), "-L", lib_dir, "-l:libpt.so", "-Xlinker", "-rpath",
           "-Xlinker", lib_dir]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return exe
