"""The first pass's warp queues and the map's device queue: where a larger
triangle is apportioned (second pass, or in the first pass when the queue is
absent or full) must not change the map, bit for bit, whatever the width of
the last strip of cells and however many triangles a row of cells adds."""
import numpy as np
import pytest

import paper_2506_02114_gb300 as mm
import synthetic
from _metrics import MAP_P999_TOL, MEAN_TOL, band_errors

pytestmark = pytest.mark.gpu

# close to critical in y: nearly every triangle of a row is a larger one, so a
# row adds up to 62 to a queue; and an ordinary model with every kind
MODELS = {"slivers": (0.8, 0.17, 0.0, 4.0), "mixed": (0.45, 0.3, 0.4, 10.0)}


@pytest.mark.parametrize("cols", [1, 30, 31, 32, 95])
@pytest.mark.parametrize("model", sorted(MODELS))
def test_queue_capacity_does_not_change_the_map(oracle_mod, model, cols):
    import torch
    torch.cuda.init()
    kappa, gamma, s, rpp = MODELS[model]
    m, pos = synthetic.star_field(11, 120, 16.0, synthetic.SALPETER_01_1)
    rows = 700
    half = (0.5 * cols * 0.05, 0.5 * rows * 0.02)
    maps, counts = [], []
    for slots in (0, -1, 1, 33, 1000):
        h = mm.create(kappa, gamma, s, m, pos, 1.0, 40, fmm_order=25, img_half=half,
                      ray_grid=(cols + 1, rows + 1), big_queue_slots=slots)
        mm.run(h, 0)
        maps.append(mm.get_map_fixed(h))
        st = mm.get_stats(h)
        assert st["error_bits"] == 0
        counts.append([st[k] for k in st if k.startswith("triangles_")])
        if slots == 0:
            mu = mm.get_map(h)
        mm.destroy(h)
    assert maps[0].any()
    for k in range(1, len(maps)):
        assert np.array_equal(maps[0], maps[k]) and counts[0] == counts[k]
    p = oracle_mod.derive_params(kappa, gamma, s, m, 1.0, 40, img_half=half,
                                 ray_grid=(cols + 1, rows + 1))
    mu_ref, _ = oracle_mod.magnification_map(p, m, pos)
    e = band_errors(mu, mu_ref, p.mu_macro)
    assert e["p999"] <= MAP_P999_TOL and (cols < 30 or e["mean_rel"] <= MEAN_TOL), e


@pytest.mark.parametrize("cols,rows", [(1, 1), (1, 700), (31, 5), (62, 63), (95, 2000)])
def test_stored_vertices_map_like_the_oracle(oracle_mod, cols, rows):
    """The plain FP64 path's mapping kernel: work items of 2 to 64 rows, the
    last strip and the last item of any width, queues kept from item to item."""
    import torch
    torch.cuda.init()
    kappa, gamma, s, _ = MODELS["mixed"]
    m, pos = synthetic.star_field(12, 60, 12.0, synthetic.SALPETER_01_1)
    half = (0.02 * cols + 0.01, 0.005 * rows + 0.01)
    grid = dict(img_half=half, ray_grid=(cols + 1, rows + 1))
    h = mm.create(kappa, gamma, s, m, pos, 2.0, 40, mode=mm.MM_PLAIN_FP64, **grid)
    mm.run(h, 0)
    mu, st = mm.get_map(h), mm.get_stats(h)
    mm.destroy(h)
    p = oracle_mod.derive_params(kappa, gamma, s, m, 2.0, 40, **grid)
    mu_ref, info = oracle_mod.magnification_map(p, m, pos)
    assert st["triangles_dropped"] == info["dropped"]
    e = band_errors(mu, mu_ref, p.mu_macro)
    assert e["p999"] <= MAP_P999_TOL, e
    # (a mean over a few cells is their outline's, to FP32)
    assert cols * rows < 1000 or e["mean_rel"] <= MEAN_TOL, e


@pytest.mark.parametrize("shape,grid,gamma,slots", [
    ((2200, 2200), (350, 300), 0.3, (0, 1000, 1 << 22)),  # too few cells for a queue by default
    ((2200, 2200), (3400, 3300), 0.3, (0, 1 << 22)),      # 2^22 slots: several first passes
    ((60, 110000), (200, 900), 0.3, (1 << 22,)),          # over a hundred bands of a narrow map
    ((30000, 300), (900, 200), 0.3, (1 << 22,)),          # 32 rows a band, triangles over many
    ((2200, 2200), (2500000, 3), -0.3, (1 << 22,)),       # more bands a triangle than there is room
])
@pytest.mark.parametrize("mode", [mm.MM_FMM_FP32, mm.MM_PLAIN_FP64])
def test_bands_of_a_large_map_do_not_change_it(shape, grid, gamma, slots, mode):
    """A map above half the L2: its second pass takes a queue of 2^22 slots or
    more by bands of rows.  Queue or none, one first pass or several, whole, in
    two rectangles of cells or in a batch: one map, bit for bit, and the same
    counts."""
    import torch
    torch.cuda.init()
    if mode == mm.MM_PLAIN_FP64 and grid[0] * grid[1] > 1000000:
        pytest.skip("the segments are the FMM path's")
    kappa, s = 0.45, 0.4
    m, pos = synthetic.star_field(13, 40, 14.0, synthetic.SALPETER_01_1)
    half = 2.0 * shape[0] / max(shape)
    opts = dict(fmm_order=20, img_half=(7.0, 3.0), ray_grid=(grid[0] + 1, grid[1] + 1),
                npix_y=shape[1], mode=mode)

    def result(h):
        st = mm.get_stats(h)
        assert st["error_bits"] == 0
        return mm.get_map_fixed(h), [st[k] for k in st if k.startswith("triangles_")], st

    def make(n):
        return mm.create(kappa, gamma, s, m, pos, half, shape[0], big_queue_slots=n, **opts)

    h = make(-1)
    mm.run(h, 0)
    ref, counts, st0 = result(h)
    mm.destroy(h)
    assert ref.any() and st0["triangles_box"] + st0["triangles_rows"] > 500
    for n in slots:
        h = make(n)
        for rep in range(2):
            mm.run(h, 0)
            got, c, st = result(h)
            assert np.array_equal(ref, got) and c == counts
        few = grid[0] * grid[1] < 1 << 21
        assert (st["queue_slots"] > 0) == (n > 0 or not few)
        if n == 1 << 22 and not few:
            assert st["kernel_launches"] > st0["kernel_launches"] + 6
        cut = grid[1] // 3
        mm.run_cells(h, 0, cut, 0, grid[0], 0)
        tot = mm.get_map_fixed(h)
        mm.run_cells(h, cut, grid[1], 0, grid[0], 0)
        assert np.array_equal(ref, tot + mm.get_map_fixed(h))
        if mode == mm.MM_FMM_FP32:
            other = make(n)
            mm.run_batch([h, other], 0)
            for one in (h, other):
                got, c, _ = result(one)
                assert np.array_equal(ref, got) and c == counts
            mm.destroy(other)
        mm.destroy(h)


@pytest.mark.parametrize("cols,rows", [(1, 3), (60, 200), (300, 900), (700, 2400), (1200, 4000),
                                       (1200, 9000)])
@pytest.mark.parametrize("model", sorted(MODELS))
def test_short_items_and_small_batches_leave_the_map_unchanged(model, cols, rows):
    """Small grids: work items of 8 to 64 rows, a second pass in batches of 4 to
    32 triangles, and with few rays per pixel a queue sized by the pixels: the
    map of long items without a queue, bit for bit."""
    import torch
    torch.cuda.init()
    kappa, gamma, s, _ = MODELS[model]
    m, pos = synthetic.star_field(14, 60, 14.0, synthetic.SALPETER_01_1)
    maps, counts = [], []
    for opts in (dict(rows_per_item=256, big_queue_slots=-1), dict(), dict(big_queue_slots=5000)):
        h = mm.create(kappa, gamma, s, m, pos, 1.5, 150, fmm_order=20, img_half=(6.0, 3.0),
                      ray_grid=(cols + 1, rows + 1), **opts)
        mm.run(h, 0)
        st = mm.get_stats(h)
        assert st["error_bits"] == 0
        maps.append(mm.get_map_fixed(h))
        counts.append([st[k] for k in st if k.startswith("triangles_")])
        mm.destroy(h)
    assert maps[0].any()
    for k in (1, 2):
        assert np.array_equal(maps[0], maps[k]) and counts[0] == counts[k]
