"""|m| of the power spectrum's modes, computed from an fp32 square root: the fp64 square root of every
m^2 that a mesh can have, to the last bit.  No GPU: the function the kernel calls, compiled for the host."""
import ctypes
import os
import subprocess

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1608_00802_gb300", "csrc")


def test_mode_norm_is_the_fp64_square_root(tmp_path):
    src = tmp_path / "mode_norm.cpp"
    src.write_text('#include "pm_mode.h"\n'
                   'extern "C" void mode_norms(double* out, uint32_t n) {\n'
                   '  for (uint32_t m2 = 1; m2 <= n; ++m2) out[m2 - 1] = pm::mode_norm(m2, sqrtf(float(m2)));\n}\n')
    lib = tmp_path / "mode_norm.so"
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)], check=True)
    n = 3 * 512 ** 2  # the corner of the largest mesh, 1024^3
    out = np.empty(n)
    ctypes.CDLL(str(lib)).mode_norms(out.ctypes.data_as(ctypes.c_void_p), ctypes.c_uint32(n))
    assert np.array_equal(out, np.sqrt(np.arange(1, n + 1, dtype=np.float64)))
