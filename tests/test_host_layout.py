"""Shared-memory layout of k_primal (CPU): every plan requests what its blocks address.

A block of `rows` rows with H halo rows keeps a table of (rows + 2H)(2H + 1) row offsets, then, from the
next 16-byte boundary (rows are read as 16-byte vectors), its rows of U with their halos."""
import ctypes
import shutil

import pytest

import fake_runtime as F

SCRIPT = """
import ctypes, json
limit, sm = 232448 - 1024, ctypes.c_int()
plans = []
for elem in (4, 8):
    for nc, H in ((1, 1), (2, 1), (1, 2)):
        for lx in range(4, 14):
            for rows in range(2, 17, 2):
                for ny in (64, 2048):
                    if lib.fake_plan_band(elem, 1 << lx, ny, nc, H, rows, limit, ctypes.byref(sm)):
                        plans.append((elem, nc, H, 1 << lx, ny, rows, sm.value))
print(json.dumps(plans))
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_primal_blocks_request_every_byte_they_address(tmp_path):
    import json
    plans = json.loads(F.run(F.build(str(tmp_path / "fake.so")), SCRIPT).splitlines()[-1])
    assert len(plans) > 300
    assert {(p[0], p[1], p[2]) for p in plans} == {(e, c, h) for e in (4, 8) for c, h in ((1, 1), (2, 1), (1, 2))}
    bad = []
    for elem, nc, H, nx, ny, rows, smem in plans:
        table = -(-(rows + 2 * H) * (2 * H + 1) * 4 // 16) * 16
        end = table + nc * (rows + 2 * H) * nx * elem
        if smem < end:
            bad.append((elem, nc, H, nx, ny, rows, smem, end))
    assert not bad, bad[:5]
