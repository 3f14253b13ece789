"""div_range over every range a scan can divide, down to 2^-60 (a noisy range can
cancel that far), for maximum ranges at and between the ends of its domain."""

import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2305_04180_gb300 import build
from tests.test_scan_math import SRC


@pytest.mark.gpu
def test_range_division_equals_ieee_down_to_the_smallest(tmp_path):
    src, lib = tmp_path / "m.cu", tmp_path / "libm.so"
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-fmad=false", "-Xcompiler", "-fPIC",
                    "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC, "-shared", str(src), "-o", str(lib)],
                   check=True)
    run = C.CDLL(str(lib)).run
    for rm in (100.0, 99.99999, 2.0 ** -20, 3.0e-5, 0.3, 366.7, 12345.678, float(np.nextafter(np.float32(2 ** 20), 0)),
               2.0 ** 20):
        rm = np.array([rm], np.float32)
        out = np.zeros(3, np.uint64)
        lo = 2.0 ** -60 / float(rm[0])
        rc = run(rm.ctypes.data_as(C.c_void_p), C.c_int(1), C.c_float(lo), out.ctypes.data_as(C.c_void_p))
        assert rc == 0 and out.tolist() == [0, 0, 0], (rm, out)
