"""The tuner's choice of a column width (CPU), on a runtime whose clock is the test's: what it measures is what the
solver then runs."""
import shutil

import pytest

import fake_runtime as F

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")

SCRIPT = """
from paper_2305_03945_gb300 import workloads as WL
lib.fake_cost(b"k_fcol", %g)
lib.fake_cost(b"k_fcol_tma", %g)
pb = WL.Problem(nx=512, ny=%d, lx=1.0, ly=4.0, bc="periodic", op="laplacian", kind="allen_cahn", dt=1e-3, a=0.05, b=20.0,
                tol=1e-11, tol_kind="f_rel")
s = rd.Solver(pb, precision="fp32_dc", autotune=1, stream=0)
cols = [n for n in F.names(lib.fake_launched) if "k_fcol" in n]
print("RUNS", "tma" if "k_fcol_tma" in cols[-1] else "threads", s.stats()["plan_col_width"])
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return F.build(str(tmp_path_factory.mktemp("fake") / "fake.so"))


@pytest.mark.parametrize("ny,threads,tma,runs", [(2048, 1.0, 0.5, "tma"), (2048, 1.0, 2.0, "threads"),
                                                 (1024, 1.0, 0.5, "threads")])
def test_column_widths_are_timed_on_the_kernel_that_runs(lib, ny, threads, tma, runs):
    out = F.run(lib, SCRIPT % (threads, tma, ny)).split()
    assert out[-2] == runs, out
    if runs == "tma":  # (a tile of less than 16-byte rows has no tensor map)
        assert int(out[-1]) >= 4


@pytest.mark.parametrize("nx,ny,width", [(16, 1024, 2), (64, 512, 2), (256, 1024, 2), (512, 512, 4), (1024, 1024, 4), (16, 64, 4)])
def test_fp64_columns_spread_over_the_chip(lib, nx, ny, width):
    """Pairs of columns while twice the blocks still fit one wave and a block keeps a warp; else 32-byte segments."""
    out = F.run(lib, """
from paper_2305_03945_gb300 import workloads as WL
pb = WL.Problem(nx=%d, ny=%d, lx=1.0, ly=1.0, bc="neumann", op="laplacian", kind="allen_cahn", dt=1e-3, a=0.05, b=20.0,
                tol=1e-11, tol_kind="f_rel")
print("WIDTH", rd.Solver(pb, stream=0).stats()["plan_col_width"])
""" % (nx, ny)).split()
    assert out[-2:] == ["WIDTH", str(width)], out
