"""The twiddles of a radix-16 pass carry no more rounding than those of a radix-8 pass.

With u = 2^-24, a table entry is off by at most u / sqrt(2) (each component rounded), by 0.41 u in the root mean
square of evenly spread rounding, and a complex product adds errors of the same kind: products of three entries, the
most a radix-8 pass multiplies, measure 0.85 to 0.92 u over a line's steps, products of four 1.02 to 1.09 u.  The
line between them is 0.97 u."""
import ctypes
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
    out = str(tmp_path_factory.mktemp("twiddle") / "probe.so")
    cmd = [B._nvcc(), *B.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", B.CSRC, "-o", out,
           os.path.join(ROOT, "tests", "twiddle_probe.cu")]
    r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    assert r.returncode == 0, r.stdout.decode()
    return ctypes.CDLL(out)


@pytest.mark.parametrize("n", [512, 1024, 2048, 4096, 8192])
def test_twiddles_of_a_radix_16_pass(probe, n):
    ang = -2.0 * np.pi * np.arange(n) / n
    tw = np.stack([np.cos(ang), np.sin(ang)], axis=-1).astype(np.float32)
    out = np.zeros((n // 16, 16, 2), np.float32)
    vp = ctypes.c_void_p
    assert probe.twiddle_probe(n, tw.ctypes.data_as(vp), out.ctypes.data_as(vp)) == 0
    step = np.arange(n // 16)[:, None] * np.arange(16)[None, :]
    err = np.abs(out[..., 0].astype(np.float64) + 1j * out[..., 1] - np.exp(-2j * np.pi * step / n))[:, 1:]
    rms = np.sqrt((err ** 2).mean(axis=0)) * 2.0 ** 24
    assert rms.max() <= 0.97, rms
