"""The library's host code on a stand-in for the CUDA runtime (fake_cudart.cpp,
no GPU): buffers are given back only after every stream that may use them, and
the pool does not keep the queues of many large maps; and the default size of
the second pass's queue, as the header states it."""
import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest

import paper_2506_02114_gb300 as mm
from paper_2506_02114_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    """libmm.so's objects linked over the stand-in, bound like the real library."""
    build.build()
    out = str(tmp_path_factory.mktemp("fake") / "libmm_fake.so")
    objs = sorted(glob.glob(os.path.join(build.OUT_DIR, "*.o")))
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", include, "-o", out,
                    os.path.join(HERE, "fake_cudart.cpp")] + objs + ["-Wl,-Bsymbolic", "-Wl,-z,defs"],
                   check=True)
    L = ctypes.CDLL(out)
    L.fake_fail_malloc.argtypes = L.fake_fail_launch.argtypes = [ctypes.c_long]
    L.fake_others.argtypes = [ctypes.c_size_t]
    for f in ("fake_unordered", "fake_mallocs", "fake_launches", "fake_pool_idle",
              "fake_total_memory"):
        getattr(L, f).restype = ctypes.c_long
    path, real = build.LIB, mm._lib
    mm._lib, build.LIB = None, out
    try:
        mm.lib(build_if_missing=False)
        yield L
    finally:
        mm._lib, build.LIB = real, path


def make(mode=mm.MM_FMM_FP32, npix=16, **more):
    pos = np.array([[0.3, 0.2], [-0.7, 0.4], [0.1, -0.6]])
    more.setdefault("ray_grid", (40, 40))
    return mm.create(0.4, 0.3, 0.0, np.ones(3), pos, 1.0, npix, mode=mode, fmm_order=4,
                     img_half=(2.0, 2.0), **more)


MODES = [mm.MM_FMM_FP32, mm.MM_PLAIN_FP64, mm.MM_FMM_IRS]


@pytest.mark.parametrize("stream", [0, 77])
@pytest.mark.parametrize("mode", MODES)
def test_destroy_waits_for_the_last_run(fake, mode, stream):
    """The default stream (NULL) is a stream like any other: a run queued
    there and never read back has to end before its buffers go back."""
    fake.fake_reset()
    h = make(mode)
    mm.run(h, stream)
    mm.run(h, stream)
    mm.destroy(h)
    assert fake.fake_unordered() == 0
    fake.fake_reset()
    h = make(mode)
    mm.run_cells(h, 0, 7, 0, 9, stream)
    mm.destroy(h)
    assert fake.fake_unordered() == 0


@pytest.mark.parametrize("mode", MODES)
def test_buffers_are_used_in_the_order_they_were_taken(fake, mode):
    """A block of the pool is there in the order of the stream it was taken
    on: until then it may be another handle's, created on another thread."""
    fake.fake_reset()
    h = make(mode)
    assert fake.fake_unordered() == 0
    mm.run(h, 0)
    mm.get_map_fixed(h)
    mm.shoot_points(h, np.zeros((3, 2)))
    mm.get_stats(h)
    assert fake.fake_unordered() == 0
    mm.destroy(h)


@pytest.mark.parametrize("stream", [0, 77])
def test_destroy_waits_for_a_batch(fake, stream):
    fake.fake_reset()
    hs = [make() for _ in range(3)]
    mm.run_batch(hs, stream)
    for h in hs:
        mm.destroy(h)
    assert fake.fake_unordered() == 0


@pytest.mark.parametrize("mode", MODES)
def test_destroy_waits_for_what_a_failed_run_queued(fake, mode):
    fake.fake_reset()
    h = make(mode)
    fake.fake_fail_launch(fake.fake_launches() + 1)   # the second of the run's
    with pytest.raises(mm.MMError):
        mm.run(h, 77)
    mm.destroy(h)
    assert fake.fake_unordered() == 0


def test_destroy_waits_for_what_a_failed_batch_queued(fake):
    """The batch's descriptor array is sized after the trees are queued."""
    fake.fake_reset()
    hs = [make() for _ in range(3)]
    fake.fake_fail_malloc(fake.fake_mallocs())
    with pytest.raises(mm.MMError) as e:
        mm.run_batch(hs, 77)
    assert e.value.status == mm.MM_ENOMEM
    for h in hs[::-1]:
        mm.destroy(h)
    assert fake.fake_unordered() == 0


def test_large_queues_do_not_stay_with_the_pool(fake):
    """One handle's queue of gigabytes may wait in the pool for the next
    handle; those of several alive at once go back."""
    fake.fake_reset()
    bound = fake.fake_total_memory() // 32
    hs = [make(npix=2200, big_queue_slots=1 << 27) for _ in range(4)]   # 5.6 GB each
    assert all(mm.get_stats(h)["queue_slots"] == 1 << 27 for h in hs)
    for h in hs[1:]:
        mm.destroy(h)
        assert fake.fake_pool_idle() <= bound
    assert fake.fake_pool_idle() > 5e9
    mm.destroy(hs[0])
    assert fake.fake_pool_idle() <= bound
    # an ordinary handle's memory stays for the next one
    idle = fake.fake_pool_idle()
    mm.destroy(make())
    assert fake.fake_pool_idle() == idle


L2, WARPS = 129 << 20, 152 * 3 * 8


def default_queue(npix, cells, kappa_star, scatter, cell, memory, mode):
    """Slots of the default queue (mm_options.big_queue_slots); scatter and a
    cell's width in pixels."""
    px = npix * npix
    if 16 * px <= L2 // 2:
        slots, ample = cells // 12, min(2 * cells, 32 * px)
        if kappa_star >= 1e-3 and slots < ample and 32 * min(ample, 1 << 27) <= memory // 32:
            slots = ample
        return min(max(slots, 1 << 16), 1 << 27)
    slots = min(2 * cells, max(cells // 5, 64 * px), 1 << 27)
    in_place = (mode == mm.MM_FMM_FP32 and scatter < 7 and cell > 1
                and cells >= 6 * WARPS * 31 * 32)
    if kappa_star < 1e-3 or slots < 1 << 22 or 42 * slots > memory // 32 or in_place:
        return 0
    return slots


@pytest.mark.parametrize("npix,n,kappa_star,scatter,cell,free_gb", [
    (100, (40, 50), 0.4, 30.0, 0.3, 270),         # the least
    (1000, (400, 300), 0.4, 30.0, 0.3, 270),      # two a cell
    (1000, (9000, 7000), 0.4, 30.0, 0.3, 270),    # 32 a pixel
    (1000, (9000, 7000), 0.4, 30.0, 0.3, 30),     #   which would leave too little
    (1000, (9000, 7000), 0.0005, 30.0, 0.3, 270),  # next to no stars: one in 12
    (1000, (60000, 50000), 0.4, 30.0, 0.3, 270),  # the most
    (2200, (350, 300), 0.4, 30.0, 0.3, 270),      # bands: too few
    (2200, (3400, 3300), 0.4, 30.0, 0.3, 270),
    (2200, (3400, 3300), 0.0005, 30.0, 0.3, 270),
    (3000, (9000, 9000), 0.4, 30.0, 0.3, 270),
    (3000, (9000, 9000), 0.4, 30.0, 0.3, 170),    # 5.6 GB would leave too little
    (2200, (5000, 5000), 0.4, 6.9, 1.01, 270),    # small stars, stretched cells: in place
    (3000, (5000, 5000), 0.4, 6.9, 1.01, 270),
    (3000, (5000, 5000), 0.4, 7.1, 1.01, 270),    # and just beyond each limit
    (3000, (5000, 5000), 0.4, 6.9, 0.99, 270),
    (3000, (4000, 5000), 0.4, 6.9, 1.01, 270),    # too few work items
])
@pytest.mark.parametrize("mode", [mm.MM_FMM_FP32, mm.MM_PLAIN_FP64])
def test_default_queue(fake, npix, n, kappa_star, scatter, cell, free_gb, mode):
    if mode == mm.MM_PLAIN_FP64 and n[0] * n[1] > 3e7:
        pytest.skip("more vertices than the path stores")
    fake.fake_reset()
    fake.fake_others(fake.fake_total_memory() - (free_gb << 30) - fake.fake_pool_idle())
    kappa, gamma = 0.4, 0.3                       # a1 = 0.9, a2 = 0.3; masses of 1
    delta = kappa_star ** 0.5 / scatter
    h = cell * delta / 0.9
    grid = dict(img_half=(0.5 * h * n[0], 0.5 * h * n[1]), ray_grid=(n[0] + 1, n[1] + 1))
    pos = np.array([[0.3, 0.2], [-0.7, 0.4], [0.1, -0.6]])
    memory = free_gb << 30

    def slots(**more):
        a = mm.create(kappa, gamma, 1.0 - kappa_star / kappa, np.ones(3), pos,
                      0.5 * delta * npix, npix, mode=mode, fmm_order=4, **grid, **more)
        try:
            return mm.get_stats(a)["queue_slots"]
        finally:
            mm.destroy(a)
            fake.fake_reset()
            fake.fake_others(fake.fake_total_memory() - memory - fake.fake_pool_idle())

    assert slots() == default_queue(npix, n[0] * n[1], kappa_star, scatter, cell, memory, mode)
    assert slots(big_queue_slots=-1) == 0
    assert slots(big_queue_slots=1 << 22) == 1 << 22
