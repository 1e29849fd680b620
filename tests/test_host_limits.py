"""Creating a solver raises the shared-memory limit (which loads the code) of the kernels it launches, and of no
others (CPU)."""
import shutil

import pytest

import fake_runtime as F

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")

SCRIPT = """
import numpy as np, ctypes
from paper_2305_03945_gb300 import workloads as WL
pb = WL.Problem(%s, lx=1.0, ly=1.0, lz=1.0, bc=%r, op=%r, kind=%r, dt=1e-3, a=0.05, b=20.0, tol=1e-11, tol_kind="f_rel"%s)
s = rd.Solver(pb, precision=%r, stream=0)
if s.precision == "fp64":
    w = np.zeros(pb.shape)
    p = ctypes.c_void_p(w.ctypes.data)
    assert lib.rd_pdhg_apply_precond(s.h, p, p) == 0, lib.rd_last_error()
print("UNUSED", sorted(set(F.names(lib.fake_limits)) - set(F.names(lib.fake_launched))))
"""

AC = ("laplacian", "allen_cahn", "")
CASES = {
    "small": ("nx=64, ny=64", "periodic", *AC, "fp32_dc"),
    "fp32": ("nx=1024, ny=128", "neumann", *AC, "fp32_dc"),
    "fp32_tma": ("nx=1024, ny=2048", "periodic", *AC, "fp32_dc"),
    "fp32_long": ("nx=4096, ny=256", "periodic", *AC, "fp32_dc"),
    "cube": ("nx=32, ny=64, nz=64", "periodic", *AC, "fp32_dc"),
    "fp64": ("nx=256, ny=128", "neumann", *AC, "fp64"),
    "two_fp64": ("nx=128, ny=128", "periodic", "laplacian", "gray_scott", ", p=(2e-3, 1e-3, 0.04, 0.06)", "fp64"),
    "ch": ("nx=256, ny=256", "periodic", "neg_biharmonic", "ch_split", "", "fp32_dc"),
    "fch": ("nx=128, ny=128", "periodic", "functionalized", "fch", "", "fp64"),
}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return F.build(str(tmp_path_factory.mktemp("fake") / "fake.so"))


@pytest.mark.parametrize("case", sorted(CASES))
def test_solver_raises_limits_of_the_kernels_it_launches(lib, case):
    out = F.run(lib, SCRIPT % CASES[case]).splitlines()[-1]
    assert out == "UNUSED []", out
