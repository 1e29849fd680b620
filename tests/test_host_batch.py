"""The batch server's host side (CPU), on a CUDA runtime in which an asynchronous copy runs as late as it may:
at the next synchronisation, reading its source then.  A graph launch finishes every step it finds begun, so
a request's result is its initial state, as far as the copies in and out are sound."""
import shutil

import pytest

import fake_runtime as F

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")

SERVE = """
import time
import numpy as np
from paper_2305_03945_gb300 import workloads as WL

def request(k, shape):
    nz, ny, nx = (1,) * (3 - len(shape)) + shape
    pb = WL.Problem(nx=nx, ny=ny, nz=nz, lx=1.0, ly=1.0, lz=1.0, bc="neumann" if k % 2 else "periodic", op="laplacian",
                    kind="allen_cahn", dt=1e-3, a=0.05, b=20.0, tol=1e-11, tol_kind="f_rel")
    return pb, WL.rng(k).standard_normal(pb.shape)

def drain(b, ids, t_max=30.0):
    got, t0 = {}, time.time()
    while len(got) < len(ids) and time.time() - t0 < t_max:
        for r in b.poll(timeout=0.2):
            got[r["id"]] = r
    return got

def serve(b, reqs):
    ids = [b.submit(pb, u0, 1, tag=k) for k, (pb, u0) in enumerate(reqs)]
    got = drain(b, ids)
    assert len(got) == len(ids), "requests that never finished"
    for (rid, out), (pb, u0) in zip(ids, reqs):
        assert got[rid]["status"] == 0, got[rid]
        assert np.array_equal(out, u0), pb.shape
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return F.build(str(tmp_path_factory.mktemp("fake") / "fake.so"))


def test_admission_keeps_its_sources_until_the_copies_have_run(lib):
    """More requests than slots (slots are used again), 2-D and 3-D, sizes on the heap and mapped."""
    F.run(lib, SERVE + """
lib.fake_slots(3)
shapes = [(64, 64), (8, 16, 16), (16, 16), (256, 512), (128, 32), (32, 32, 32), (4, 8), (512, 64)]
with rd.Batch(1 << 26, 3, stream=0) as b:
    serve(b, [request(k, s) for k, s in enumerate(shapes)])
""", env={"MALLOC_PERTURB_": "165"})


def test_serving_allocates_no_device_memory(lib):
    """With device memory exhausted once the batch is made, requests of every route are still served."""
    F.run(lib, SERVE + """
lib.fake_slots(4)
with rd.Batch(1 << 28, 4, stream=0) as b:
    serve(b, [request(0, (64, 64))])
    lib.fake_refuse_alloc(1)
    n = lib.fake_alloc_calls()
    shapes = [(1024, 1024), (512, 1024), (1024, 4), (4, 1024), (128, 128), (16, 16), (4, 4), (64, 64, 64), (4, 32, 32), (16, 512, 16)]
    serve(b, [request(k, s) for k, s in enumerate(shapes)])
    serve(b, [request(k, (1024, 1024)) for k in range(8)])
    assert lib.fake_alloc_calls() == n
    lib.fake_refuse_alloc(0)
""")


@pytest.mark.parametrize("length", [6.58562070071191, 0.9680646812275848, 5.784860330543764, 1.0])
def test_eigenvalues_are_rounded_once(lib, length):
    """The FP32 eigenvalues of a slot are the long double ones rounded: on the first three lengths, rounding them to
    double on the way changes one of them."""
    F.run(lib, SERVE + """
import ctypes
L = np.longdouble
length, n = %r, 1024
lib.fake_slots(1)
with rd.Batch(1 << 25, 1, stream=0) as b:
    pb, u0 = request(1, (16, n))
    serve(b, [(pb.replace(lx=length), u0)])
    h = L(length / n)
    sn = np.sin(L("3.141592653589793238462643383279502884") * np.arange(n).astype(L) / L(2 * n))
    mu = (L(4) / (h * h) * sn * sn).astype(np.float32)
    lib.fake_contains.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
    assert lib.fake_contains(mu.ctypes.data, mu.nbytes) == 1
""" % length)


def test_small_solves_alone_fill_a_longer_graph(lib):
    """Inner solves per graph of the one-launch slots: half of graph_k alone, a quarter beside other branches."""
    F.run(lib, SERVE + """
lib.fake_slots(4)
def solves():
    return sum("k_small" in n for n in F.names(lib.fake_launched))
with rd.Batch(1 << 26, 4, graph_k=16, stream=0) as b:
    serve(b, [request(0, (4, 4))])
    assert solves() == 8, solves()
with rd.Batch(1 << 26, 4, graph_k=16, stream=0) as b:
    n, ids = solves(), []
    lib.fake_hold(1)
    for k, s in enumerate([(256, 256), (4, 4)]):  # the second joins the first, still running
        ids.append(b.submit(*request(k, s), 1))
        t0 = time.time()
        while b.stats()["admitted"] < k + 1 and time.time() - t0 < 30:
            time.sleep(0.01)
    lib.fake_hold(0)
    assert len(drain(b, ids)) == 2
    assert solves() - n == 4, solves() - n
""")
