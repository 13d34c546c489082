"""The library's host code on a stand-in for the CUDA runtime (fake_cudart.cpp,
no GPU): buffers are given back only after every stream that may use them, and
the pool does not keep the queues of many large maps."""
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
    handle; those of several alive at once go back to the driver."""
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
