"""The batched line kernels (rd_batch_lines.cuh) at the edges of their ranges: every line length,
uneven sides, both boundaries, one and two components, 2-D and 3-D, several slots of different sizes in
one launch, more line groups than blocks; and sides below 16 points beside them.

Tolerance: 1e-9 relative per run of one or two steps solved to 1e-11, as everywhere in the suite.
"""
import time

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


def _req(k, kind, bc, ny, nx, nz=1):
    op = "neg_biharmonic" if kind.startswith("ch") else "laplacian"
    h = 1.0 / 64
    p = {"gray_scott": (2e-3, 1e-3, 0.04, 0.06), "schnakenberg": (0.05, 1.0, 100.0, 0.1305, 0.7695)}.get(kind, ())
    pb = WL.Problem(nx=nx, ny=ny, nz=nz, lx=h * nx, ly=h * ny, lz=h * nz, bc=bc, op=op, kind=kind, p=p,
                    dt={"gray_scott": 0.5, "schnakenberg": 2e-4}.get(kind, 1e-5 if op != "laplacian" else 2e-3),
                    a=4e-4 if op != "laplacian" else 0.05, b=1.0 if op != "laplacian" else 20.0, tau_u=0.9,
                    tau_p=0.9, tol=1e-11, tol_kind="f_rel")
    u0 = WL.uniform_field(90 + k, pb.shape, 0.4, 0.6) if pb.ncomp == 2 else WL.uniform_field(90 + k, pb.shape, -0.5, 0.5)
    return pb, u0, 1 + k % 2


MIXES = {
    "2d": [("allen_cahn", "periodic", 16, 16), ("allen_cahn", "neumann", 1024, 16), ("allen_cahn", "periodic", 16, 1024),
           ("ch_split", "neumann", 32, 512), ("ch_implicit", "periodic", 256, 64), ("none", "neumann", 64, 128),
           ("allen_cahn", "neumann", 1024, 1024), ("ch_split", "periodic", 8, 256)],
    "two_species": [("gray_scott", "periodic", 16, 32), ("gray_scott", "neumann", 32, 1024), ("schnakenberg", "neumann", 128, 64)],
    "3d": [("allen_cahn", "periodic", 16, 16, 16), ("ch_split", "neumann", 64, 16, 32), ("allen_cahn", "neumann", 16, 128, 16),
           ("ch_implicit", "periodic", 32, 16, 128), ("allen_cahn", "periodic", 16, 256, 16), ("allen_cahn", "neumann", 8, 32, 64)],
}


@pytest.mark.parametrize("mix", sorted(MIXES))
def test_line_kernels_match_oracle_in_a_mix(mix):
    from paper_2305_03945_gb300 import rd
    reqs = [_req(k, *m) for k, m in enumerate(MIXES[mix])]
    results = {}
    with rd.Batch(1 << 30, 16, small_solve=0) as b:
        ids = [b.submit(pb, u0, n, tag=k) for k, (pb, u0, n) in enumerate(reqs)]
        t0 = time.time()
        while len(results) < len(ids) and time.time() - t0 < 120:
            for r in b.poll(timeout=1.0):
                results[r["id"]] = r
    assert len(results) == len(reqs)
    for (rid, out), (pb, u0, n) in zip(ids, reqs):
        assert results[rid]["status"] == 0 and results[rid]["steps"] == n, results[rid]
        U, _ = O.solve(pb, u0, n)
        assert np.linalg.norm(out - U) <= 1e-9 * np.linalg.norm(U), (pb.kind, pb.bc, pb.shape)
