"""The FP32 3-D kernels on register-resident line transforms (rd_cube.cuh) at the edges of their
ranges: the shortest sides, uneven sides, both numbers of values per thread (grids below and from
2^20 points), a partly filled last block, both boundaries and stencils.

Tolerance: 1e-9 relative per defect-corrected step (solved to 1e-11), as everywhere in the suite.
"""
import numpy as np
import pytest

from oracle import rd_oracle as O
from paper_2305_03945_gb300 import workloads as WL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_03945_gb300 import build
    build.build()


@pytest.mark.parametrize("loop", ["graph", "host"])
@pytest.mark.parametrize("kind,bc,nz,ny,nx", [
    ("allen_cahn", "periodic", 16, 16, 16), ("ch_split", "neumann", 16, 16, 16), ("ch_implicit", "periodic", 16, 64, 32),
    ("allen_cahn", "neumann", 64, 16, 128), ("none", "neumann", 32, 128, 16), ("allen_cahn", "periodic", 16, 32, 256),
    ("ch_split", "periodic", 64, 128, 128), ("allen_cahn", "neumann", 256, 32, 128), ("ch_split", "neumann", 16, 256, 256)])
def test_cube_step_matches_oracle(kind, bc, nz, ny, nx, loop):
    from paper_2305_03945_gb300 import rd
    op = "neg_biharmonic" if kind.startswith("ch") else "laplacian"
    h = 1.0 / 64
    pb = WL.Problem(nx=nx, ny=ny, nz=nz, lx=h * nx, ly=h * ny, lz=h * nz, bc=bc, op=op, kind=kind,
                    dt=1e-5 if op != "laplacian" else 2e-3, a=4e-4 if op != "laplacian" else 0.05,
                    b=1.0 if op != "laplacian" else 20.0, tau_u=0.9, tau_p=0.9, tol=1e-11, tol_kind="f_rel",
                    max_iter=3000)
    uk = WL.uniform_field(5, pb.shape, -0.5, 0.5)
    with rd.Solver(pb, precision="fp32_dc", solve_loop=loop) as s:
        u = torch.from_numpy(uk).cuda()
        out = torch.empty_like(u)
        info = s.step(u, out)
    U, _ = O.pdhg_step(pb, uk)
    assert info["status"] == 0, info
    assert np.linalg.norm(out.cpu().numpy() - U) <= 1e-9 * np.linalg.norm(U)
