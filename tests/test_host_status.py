"""How a solve's device status reaches the caller (CPU): a graph of the runtime under test ends with the status the
test asks for.  A kernel whose wait ran out is a device error, never a diverged or unconverged iteration."""
import shutil

import pytest

import fake_runtime as F

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")

# rd_internal.h: StStatus
CONVERGED, NOT_CONVERGED, DIVERGED, FAULT = 1, 2, 3, 5

SCRIPT = """
import ctypes
import numpy as np
from paper_2305_03945_gb300 import workloads as WL
lib.fake_status(%d, %d)
pb = WL.Problem(nx=512, ny=2048, lx=1.0, ly=4.0, bc="periodic", op="laplacian", kind="allen_cahn", dt=1e-3, a=0.05, b=20.0,
                tol=1e-11, tol_kind="f_rel")
s = rd.Solver(pb, precision=%r, stream=0)
u, info = np.zeros(pb.shape), rd.rd_step_info()
p = ctypes.c_void_p(u.ctypes.data)
print("STATUS", lib.rd_pdhg_step(s.h, p, p, ctypes.byref(info)), info.status, lib.rd_last_error().decode())
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return F.build(str(tmp_path_factory.mktemp("fake") / "fake.so"))


@pytest.mark.parametrize("precision", ["fp32_dc", "fp64"])
@pytest.mark.parametrize("status,code", [(CONVERGED, 0), (NOT_CONVERGED, 5), (DIVERGED, 6), (FAULT, 4)])
def test_solve_status_reaches_the_caller(lib, status, code, precision):
    out = F.run(lib, SCRIPT % (status, status, precision)).splitlines()[-1].split(None, 3)
    assert out[1:3] == [str(code)] * 2, out
    assert (status == FAULT) == ("wait" in "".join(out[3:]))


def test_outer_loop_ends_with_its_inner_solves_fault(lib):
    out = F.run(lib, "print([lib.fake_outer_after_inner(k) for k in (%d, %d, %d, %d)])"
                % (CONVERGED, NOT_CONVERGED, DIVERGED, FAULT)).splitlines()[-1]
    assert out == "[0, 0, %d, %d]" % (DIVERGED, FAULT)
