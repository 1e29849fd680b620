"""The sweep kernels on register-resident line transforms (k_fcol, k_rowfwd, k_dual, k_primal) at the
edges of their ranges: every line length with either number of values per thread, ragged last
bands, the lowest grids, both boundaries, both precisions.

Tolerances: FP64 operators 1e-12 of the largest value (a transform of N points errs by a few
eps log2 N); defect-corrected steps 1e-9 (the step is solved to 1e-11), as everywhere in the suite.
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


def _pb(kind, bc, ny, nx, **kw):
    op = "neg_biharmonic" if kind.startswith("ch") else "laplacian"
    p = {"gray_scott": (2e-3, 1e-3, 0.04, 0.06), "schnakenberg": (0.05, 1.0, 100.0, 0.1305, 0.7695)}.get(kind, ())
    dt = {"gray_scott": 0.5, "schnakenberg": 2e-4}.get(kind, 1e-5 if op != "laplacian" else 2e-3)
    a, b = (4e-4, 1.0) if op != "laplacian" else (0.05, 20.0)
    # square cells no finer than 1/512: on finer ones the biharmonic term a dt / h^4 of the
    # Cahn-Hilliard states puts the FP64 residual's own rounding floor above the threshold
    lx = max(1.0, nx / 512)
    return WL.Problem(nx=nx, ny=ny, lx=lx, ly=lx * ny / nx, bc=bc, op=op, kind=kind, dt=dt, a=a, b=b, p=p,
                      tau_u=0.9, tau_p=0.9, tol=1e-11, tol_kind="f_rel", max_iter=3000)


def _state(pb, seed):
    if pb.ncomp == 2:
        return 0.5 + WL.uniform_field(seed, pb.shape, -0.1, 0.1)
    return WL.uniform_field(seed, pb.shape, -0.5, 0.5)


# every length with V = 4 (short grids) and with V = 16 (grids of 2^20 points and more)
LENGTHS = [(16, 16), (16, 2048), (2048, 16), (32, 64), (128, 32), (256, 512), (1024, 128), (2, 1024), (4, 512),
           (512, 2048), (2048, 512), (1024, 1024), (256, 4096), (4096, 256)]


@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("ny,nx", LENGTHS)
def test_preconditioner_every_line_length(ny, nx, bc):
    from paper_2305_03945_gb300 import rd
    pb = _pb("schnakenberg" if ny * nx <= 4096 else "allen_cahn" if nx == 4096 else "ch_split", bc, ny, nx)
    W = WL.rng(3).standard_normal(pb.shape)
    with rd.Solver(pb) as s:
        w = torch.from_numpy(W).cuda()
        y = torch.empty_like(w)
        s.apply_precond(w, y)
    want = O.apply_ginv(pb, W)
    assert np.max(np.abs(y.cpu().numpy() - want)) <= 1e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("precision", ["fp64", "fp32_dc"])
@pytest.mark.parametrize("kind,bc,ny,nx,rows", [
    ("allen_cahn", "neumann", 2, 64, 2), ("ch_implicit", "neumann", 4, 32, 2), ("ch_split", "periodic", 2, 16, 2),
    ("allen_cahn", "periodic", 64, 512, 6), ("ch_implicit", "periodic", 32, 256, 10), ("gray_scott", "neumann", 64, 128, 14),
    ("schnakenberg", "periodic", 16, 1024, 0), ("none", "neumann", 128, 16, 0),
    ("allen_cahn", "neumann", 1024, 1024, 0), ("ch_split", "neumann", 512, 2048, 0), ("gray_scott", "periodic", 1024, 512, 6)])
def test_step_matches_oracle_at_the_edges(kind, bc, ny, nx, rows, precision):
    """Bands that do not divide the grid, bands of the whole grid, two-row grids (whose halo wraps
    onto the band itself), V = 4 and V = 16."""
    from paper_2305_03945_gb300 import rd
    pb = _pb(kind, bc, ny, nx)
    uk = _state(pb, 4)
    with rd.Solver(pb, precision=precision, upd_rows=rows, small_solve=0) as s:
        assert s.stats()["fused_update"] == 1
        u = torch.from_numpy(uk).cuda()
        out = torch.empty_like(u)
        info = s.step(u, out)
    U, _ = O.pdhg_step(pb, uk)
    assert info["status"] == 0, info
    assert np.linalg.norm(out.cpu().numpy() - U) <= 1e-9 * np.linalg.norm(U)


@pytest.mark.parametrize("kind,bc,ny,nx", [("allen_cahn", "neumann", 2048, 512), ("gray_scott", "neumann", 2048, 512),
                                           ("ch_split", "periodic", 2048, 1024), ("allen_cahn", "neumann", 4096, 256),
                                           ("allen_cahn", "neumann", 8192, 128), ("ch_split", "periodic", 4096, 16)])
def test_columns_moved_by_tma(kind, bc, ny, nx):
    """The FP32 column solve on lines of 2048 points and more (k_fcol_tma): both boundaries, one and two
    components, the narrowest grid its tiles cover."""
    from paper_2305_03945_gb300 import rd
    pb = _pb(kind, bc, ny, nx).replace(ly=4.0, lx=4.0 * nx / ny)
    uk = _state(pb, 6)
    with rd.Solver(pb, precision="fp32_dc") as s:
        u = torch.from_numpy(uk).cuda()
        out = torch.empty_like(u)
        info = s.step(u, out)
    U, _ = O.pdhg_step(pb, uk)
    assert info["status"] == 0, info
    assert np.linalg.norm(out.cpu().numpy() - U) <= 1e-9 * np.linalg.norm(U)
