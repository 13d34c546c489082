"""Leaf records of one leaf, straight from their kernels (leaf_records.cu):
what the plan's count of direct stars and the culling bound promise."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2506_02114_gb300 import build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ERR_NEAR_SLOTS = 16
REC = np.dtype([("ref", "i4", 2), ("fc", "f4", 2), ("U", "i4", 2), ("Uf", "f4", 2), ("zs", "f4", 2),
                ("near_off", "i4"), ("near_cnt", "i4"), ("coef_off", "i4"), ("node", "i4"),
                ("cull_side", "i4"), ("cull_r2", "f4")])


@pytest.fixture(scope="module")
def records(tmp_path_factory):
    import torch
    torch.cuda.init()
    build.build()
    out = str(tmp_path_factory.mktemp("leaf") / "libleaf.so")
    subprocess.run([build.nvcc()] + build.ARCH +
                   ["-shared", "-std=c++17", "-Xcompiler", "-fPIC", "-I", build.INCLUDE, "-I",
                    build.CSRC, "--expt-relaxed-constexpr", "-o", out,
                    os.path.join(HERE, "leaf_records.cu"), os.path.join(build.OUT_DIR, "fmm.o")],
                   check=True)
    L = ctypes.CDLL(out)
    dp, up = ctypes.POINTER(ctypes.c_double), ctypes.POINTER(ctypes.c_uint)
    L.leaf_records.argtypes = [dp, dp, dp, ctypes.c_int64, ctypes.c_int, ctypes.c_int64,
                               ctypes.c_double, ctypes.c_void_p, up, up, up]

    def run(x, y, m, sub, cap, lox=-1000.0):
        a = [np.ascontiguousarray(v, dtype=np.float64) for v in (x, y, m)]
        recs = np.zeros(4 ** sub, REC)
        total, err, written = ctypes.c_uint(), ctypes.c_uint(), (ctypes.c_uint * 2)()
        e = L.leaf_records(*[v.ctypes.data_as(dp) for v in a], len(a[0]), sub, cap, lox,
                           recs.ctypes.data, ctypes.byref(total), written, ctypes.byref(err))
        assert e == 0
        return recs, total.value, list(written), err.value
    return run


@pytest.mark.parametrize("sub", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 7, 40])
def test_direct_stars_without_a_slot_are_reported(records, n, sub):
    """The plan's count is exactly what the records take; one slot less and
    the record that finds none says so and writes nothing beyond the rest."""
    rng = np.random.default_rng(100 * n + sub)
    x, y, m = 16.0 * rng.random(n) - 8.0, 16.0 * rng.random(n) - 8.0, 0.1 + rng.random(n)
    recs, total, written, err = records(x, y, m, sub, -1)
    assert err == 0 and recs["near_cnt"].sum() == total and written == [total, 0]
    recs, total, written, err = records(x, y, m, sub, -2)
    assert err == ERR_NEAR_SLOTS and written[1] == 0
    assert recs["near_cnt"].sum() < total
