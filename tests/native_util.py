"""Compiles a test's own CUDA source against the library's headers."""
import ctypes
import os
import subprocess

from paper_2110_10156_gb300 import build


def compile_shared(source, out_dir, extra=()):
    """The shared library of tests/native/<source>, path in out_dir."""
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native", source)
    out = os.path.join(str(out_dir), source.replace(".cu", ".so"))
    cmd = [build.nvcc()] + build.NVCC_FLAGS + ["-I", build.CSRC, "-shared", "-Xlinker", "-Bsymbolic", src,
                                               "-o", out, "-lcudart", *extra]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    return out


def load(source, out_dir, extra=()):
    return ctypes.CDLL(compile_shared(source, out_dir, extra))
