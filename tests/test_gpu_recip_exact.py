"""The reciprocal of the density in node pairs equals the one-node kernels'
division for every FP32 bit pattern: the ground on which both store the same
bits at any density, not only near 1."""
import ctypes
import os
import subprocess

import pytest

from gpu_common import dev
from paper_1801_04586_gb300 import builder

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_recip_exact_is_the_division(tmp_path):
    dev()
    lib = str(tmp_path / "librecip.so")
    cmd = [builder.nvcc(), *builder.ARCH, *builder.FLAGS, "-I", builder.CSRC, "-shared",
           os.path.join(HERE, "recip_exact_check.cu"), "-o", lib]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = (ctypes.c_ulonglong * 2)()
    assert ctypes.CDLL(lib).recip_exact_mismatches(out) == 0
    assert list(out) == [0, 0]
