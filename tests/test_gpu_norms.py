"""The norm that stops a solve is summed beyond FP32, whatever the arithmetic of the sweep.

The kernels sum the squares of up to 32 FP32 residuals of a line group in twice FP32's precision, off by at
most 32^2 2^-48 = 3.6e-12 of the sum, and add the groups in FP64 (a chain of less than 100 additions, 1e-14): the
norm is within 1.9e-12 of the exact one.  FP32 sums miss that by three orders of magnitude."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_03945_gb300 import build as B
    out = str(tmp_path_factory.mktemp("norm") / "probe.so")
    cmd = [B._nvcc(), *B.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", B.CSRC, "-o", out,
           os.path.join(ROOT, "tests", "norm_probe.cu")]
    r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    assert r.returncode == 0, r.stdout.decode()
    return ctypes.CDLL(out)


@pytest.mark.parametrize("which", range(4), ids=["k3_rowres", "k_primal_long", "k_rowres_b_3d", "k_rowres_b_2d"])
def test_norm_is_summed_beyond_fp32(probe, which):
    side, norm = (ctypes.c_int * 3)(), ctypes.c_double()
    assert probe.norm_probe(which, side, None, None) == 0
    n = side[0] * side[1] * side[2]
    r = np.random.default_rng(7 + which).standard_normal(n).astype(np.float32)
    assert probe.norm_probe(which, side, r.ctypes.data_as(ctypes.c_void_p), ctypes.byref(norm)) == 0
    exact = math.sqrt(math.fsum(r.astype(np.float64) ** 2))
    assert abs(norm.value - exact) <= 1.9e-12 * exact, norm.value / exact - 1
