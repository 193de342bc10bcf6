"""Compiles the small native checks of tests/native against the library."""
import os
import subprocess

from paper_1406_4350_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))


def run(name, tmp_path):
    """Build tests/native/<name>.cu, run it and return its rows of numbers."""
    lib = b.build()
    exe = str(tmp_path / name)
    src = os.path.join(HERE, "native", name + ".cu")
    r = subprocess.run([b._nvcc(), *b.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I" + b.INCLUDE,
                        "-I" + b.CSRC, src, "-o", exe, lib, "-Xlinker", "-rpath=" + os.path.dirname(lib)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    return [list(map(float, line.split())) for line in r.stdout.split("\n") if line.strip()]
