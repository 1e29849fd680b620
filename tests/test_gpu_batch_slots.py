"""Slots of a batch (GPU): the longest lines of 3-D slots along every axis, and slots that run on beside others that
were retired from under the same work lists.

Tolerance: 1e-9 relative per run of one or two steps solved to 1e-11, as everywhere in the suite; a slot's own
result does not depend on its company, bit for bit."""
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


def _req(k, kind, bc, shape):
    nz, ny, nx = (1,) * (3 - len(shape)) + shape
    ch = kind.startswith("ch")
    h = 1.0 / 64
    pb = WL.Problem(nx=nx, ny=ny, nz=nz, lx=h * nx, ly=h * ny, lz=h * nz, bc=bc, op="neg_biharmonic" if ch else "laplacian",
                    kind=kind, dt=1e-5 if ch else 2e-3, a=4e-4 if ch else 0.05, b=1.0 if ch else 20.0, tau_u=0.9, tau_p=0.9,
                    tol=1e-11, tol_kind="f_rel")
    return pb, WL.uniform_field(170 + k, pb.shape, -0.5, 0.5)


def _run(runs, slots=16):
    from paper_2305_03945_gb300 import rd
    done = {}
    with rd.Batch(1 << 30, slots) as b:
        ids = [b.submit(pb, u0, n, tag=k) for k, (pb, u0, n) in enumerate(runs)]
        t0 = time.time()
        while len(done) < len(ids) and time.time() - t0 < 120:
            for r in b.poll(timeout=1.0):
                done[r["id"]] = r
    assert len(done) == len(ids)
    assert all(done[i]["status"] == 0 and done[i]["steps"] == n for (i, _), (_, _, n) in zip(ids, runs))
    return [out for _, out in ids], [done[i]["iterations"] for i, _ in ids]


@pytest.mark.parametrize("kind,bc", [("allen_cahn", "periodic"), ("ch_split", "neumann")])
def test_longest_lines_of_a_3d_slot(kind, bc):
    reqs = [_req(k, kind, bc, s) for k, s in enumerate([(16, 16, 512), (16, 512, 16), (512, 16, 16)])]
    outs, _ = _run([(pb, u0, 1) for pb, u0 in reqs])
    for out, (pb, u0) in zip(outs, reqs):
        U, _ = O.solve(pb, u0, 1)
        assert np.linalg.norm(out - U) <= 1e-9 * np.linalg.norm(U), pb.shape


@pytest.mark.parametrize("shape", [(64, 64), (256, 128), (8, 64), (32, 32, 32), (8, 16, 16)])
def test_a_slot_runs_on_beside_retired_ones(shape):
    """One long run among short ones of its kind, which leave while it runs; some are admitted into slots that others
    left."""
    long_run = _req(0, "allen_cahn", "neumann", shape)
    short = [_req(1 + k, "allen_cahn", "periodic" if k % 2 else "neumann", s)
             for k, s in enumerate([shape, (16, 16), (128, 64), (16, 16, 16), shape, (64, 128), (4, 16), shape])]
    runs = [(*long_run, 12)] + [(pb, u0, 1 + k % 3) for k, (pb, u0) in enumerate(short)]
    outs, its = _run(runs, slots=6)
    alone, it = _run([(*long_run, 12)])
    assert np.array_equal(outs[0], alone[0]) and its[0] == it[0]
