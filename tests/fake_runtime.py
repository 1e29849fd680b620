"""Builds the library's objects against tests/fake_cudart.cpp, so that its host code runs without a GPU.

``load(tmp)`` runs in a child process (the library must not be loaded twice in one) and returns the
``rd`` module bound to that build, and the library.  Never a test of a kernel: none runs.
"""
import ctypes
import glob
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def build(out):
    from paper_2305_03945_gb300 import build as B
    B.build()
    objs = [os.path.join(B.BUILD, os.path.basename(s).replace(".cu", ".o")) for s in B._sources()]
    if not all(os.path.exists(o) for o in objs):
        B.build(force=True)
    cuda = os.path.dirname(os.path.dirname(B._nvcc()))
    inc = [p for p in (os.path.join(cuda, "include"), *glob.glob(os.path.join(cuda, "targets", "*", "include")))
           if os.path.exists(p)]
    cmd = ["g++", "-std=c++17", "-O1", "-g", "-shared", "-fPIC", "-o", out, os.path.join(ROOT, "tests", "fake_cudart.cpp"),
           *objs, "-I", B.CSRC, *[a for p in inc for a in ("-I", p)], "-lpthread",
           "-Wl,--no-undefined", "-Wl,-Bsymbolic"]  # its own runtime, whatever else the process has loaded
    r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    if r.returncode:
        raise RuntimeError(r.stdout.decode(errors="replace"))
    return out


def load(path):
    from paper_2305_03945_gb300 import rd
    lib = rd.load(path)
    lib.fake_alloc_calls.restype = ctypes.c_long
    lib.fake_launched.restype = lib.fake_limits.restype = ctypes.c_size_t
    lib.fake_slots.argtypes = [ctypes.c_size_t]
    lib.fake_launched.argtypes = lib.fake_limits.argtypes = [ctypes.c_char_p, ctypes.c_size_t]
    lib.fake_cost.argtypes = [ctypes.c_char_p, ctypes.c_float]
    return rd, lib


def names(fn):
    n = fn(None, 0)
    buf = ctypes.create_string_buffer(n)
    fn(buf, n)
    return buf.value.decode().split("\n")[:-1]


def run(path, script, timeout=300, env=None):
    """Runs ``script`` in a child process whose ``rd`` and ``lib`` are this build's; returns its output."""
    head = ("import sys; sys.path.insert(0, %r); sys.path.insert(0, %r)\n"
            "import fake_runtime as F\nrd, lib = F.load(%r)\n" % (ROOT, os.path.join(ROOT, "tests"), path))
    r = subprocess.run([sys.executable, "-c", head + script], stdout=subprocess.PIPE, stderr=subprocess.STDOUT,
                       timeout=timeout, cwd=ROOT, env={**os.environ, **(env or {})})
    out = r.stdout.decode(errors="replace")
    assert r.returncode == 0, out
    return out
