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


@pytest.mark.parametrize("n,mass", [(1, 0.7), (300, 0.3), (4000000, 1.0155)])
def test_culling_radius_covers_the_direct_mass(records, n, mass):
    """Beyond the radius the direct stars' whole mass moves a vertex by less
    than the record's distance from the map (1000 - 8 - 16 pixels: the centre's
    image, the macro term over the leaf, the map) less the margin of 2.  Millions
    of stars in one place: in FP32 each would add its mass rounded to the sum's
    last bit (1/32 here, a loss of 1.5 % a star)."""
    recs, total, _, err = records(np.full(n, 0.3), np.full(n, -0.2), np.full(n, mass), 0, -1)
    assert err == 0 and total == n and recs["near_cnt"][0] == n
    side = recs["cull_side"][0]
    assert side == 2   # beyond the right edge
    # |1 - kappa + kappa_* + gamma| (L + h) / delta, with h = 0.5 and L = 8
    D = 1000.0 - 1.3 * 8.5 - 16.0
    r2 = (n * mass / (D - 2.0) / 0.5) ** 2
    assert r2 <= recs["cull_r2"][0] <= 1.02 * r2
