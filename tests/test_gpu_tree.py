"""The quadtree built on the device against the split rule applied on the
host, and the expansions' translations at the orders where their work is
dealt out differently."""
import math

import numpy as np
import pytest

import paper_2506_02114_gb300 as mm
import synthetic
from _metrics import DEFLECTION_TOL, deflection_rel_error

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()


def host_tree(pos, R0, limit):
    """(nodes per level, leaves) of the tree: a node splits when the stars in
    its 3 x 3 block of same-level cells exceed the limit, down to level 21."""
    cell = np.clip(np.floor((pos + R0) * ((1 << 21) / (2.0 * R0))), 0, (1 << 21) - 1).astype(np.int64)
    nodes, counts, leaves = {(0, 0)}, [], 0
    for level in range(22):
        counts.append(len(nodes))
        c = cell >> (21 - level)
        n = {}
        for x, y in c.tolist():
            n[x, y] = n.get((x, y), 0) + 1
        nxt = set()
        for x, y in nodes:
            block = sum(n.get((x + dx, y + dy), 0) for dx in (-1, 0, 1) for dy in (-1, 0, 1))
            if level < 21 and block > limit:
                nxt |= {(2 * x + i, 2 * y + j) for i in (0, 1) for j in (0, 1)}
            else:
                leaves += 1
        nodes = nxt
        if not nodes:
            break
    return counts, leaves


def fields():
    u = synthetic.uniform
    disk = synthetic.star_field(5, 9000, 40.0, synthetic.EQUAL)[1]
    yield "one", np.array([[0.3, -0.2]]), 1
    yield "pair at one place", np.array([[0.7, 0.7], [0.7, 0.7], [-3.0, 2.0]]), 1   # depth 21
    yield "few", disk[:33] * 0.1, 32
    yield "9000, levels above 1024 nodes", disk, 8
    yield "9000, leaf size 1", disk[:3000], 1
    # a dense clump in a sparse field: neighbours many levels coarser
    clump = np.stack([2.0 + 1e-3 * u(3, 0, 2000), 1.0 + 1e-3 * u(3, 1, 2000)], 1)
    yield "clump", np.concatenate([disk[:500], clump]), 16
    yield "line", np.stack([40.0 * u(4, 0, 4000) - 20.0, np.zeros(4000)], 1), 20


@pytest.mark.parametrize("name", [f[0] for f in fields()])
def test_tree_follows_the_split_rule(name):
    _, pos, limit = next(f for f in fields() if f[0] == name)
    h = mm.create(0.4, 0.3, 0.0, np.ones(len(pos)), pos, 1.0, 16, fmm_order=4, leaf_size=limit,
                  img_half=(2.0, 2.0), ray_grid=(40, 40))
    for _ in range(2):   # the plan's tree, then the run's
        st = mm.get_stats(h)
        counts, leaves = host_tree(pos, st["root_half_length"], limit)
        assert (st["nodes"], st["leaves"], st["depth"]) == (sum(counts), leaves, len(counts) - 1)
        assert st["error_bits"] == 0
        mm.run(h, 0)
        mm.run(h, 0)
    mm.destroy(h)


@pytest.mark.parametrize("p", [1, 2, 3, 20, 31, 32, 33, 40, 63, 64])
@pytest.mark.parametrize("leaf", [4, 100])
@pytest.mark.parametrize("sub", [-1, 1, 2])
def test_deflection_at_every_dealing_of_the_order(oracle_mod, p, leaf, sub):
    """Worst case of the truncated translations: a source's multipole at the
    nearest well-separated cell converges like r = sqrt(2) / (4 - sqrt(2)), so
    the deflection's error is at most a few times r^p of the deflection (the
    leading coefficient 1 / (1 - r) = 2.2 for the potential, times p + 1 for
    its derivative), on top of the FP32 evaluation.  The sub-cells' series are
    cut where their own bound, (sqrt(2) / 3)^p, is below that."""
    m, pos = synthetic.star_field(17, 700, 30.0, synthetic.SALPETER_01_1)
    kappa, gamma, s = 0.4, 0.3, 0.2
    grid = dict(img_half=(6.0, 6.0), ray_grid=(241, 241))
    h = mm.create(kappa, gamma, s, m, pos, 1.0, 16, fmm_order=p, leaf_size=leaf, sub_levels=sub,
                  **grid)
    z = 12.0 * np.stack([synthetic.uniform(8, 0, 2000), synthetic.uniform(8, 1, 2000)], 1) - 6.0
    w = mm.shoot_points(h, z)
    mm.destroy(h)
    par = oracle_mod.derive_params(kappa, gamma, s, m, 1.0, 16, **grid)
    w_ref = oracle_mod.deflect(par, m, pos, z)
    r = math.sqrt(2.0) / (4.0 - math.sqrt(2.0))
    err = deflection_rel_error(par, z, w, w_ref).max()
    assert err <= DEFLECTION_TOL + 2.2 * (p + 1) * r ** p, err


def test_probe_buffer_of_any_size():
    """Source positions do not depend on the calls before: small, large (given
    back) and small again, on both paths."""
    m, pos = synthetic.star_field(17, 100, 12.0, synthetic.EQUAL)
    n = (1 << 20) + 3
    z = 4.0 * np.stack([synthetic.uniform(9, 0, n), synthetic.uniform(9, 1, n)], 1) - 2.0
    for mode in (mm.MM_FMM_FP32, mm.MM_PLAIN_FP64):
        h = mm.create(0.4, 0.3, 0.0, m, pos, 1.0, 16, fmm_order=20, mode=mode, img_half=(2.0, 2.0),
                      ray_grid=(101, 101))
        few = mm.shoot_points(h, z[:7])
        whole = mm.shoot_points(h, z)
        assert np.array_equal(whole[:7], few) and np.isfinite(whole).all()
        assert np.array_equal(mm.shoot_points(h, z[-5:]), whole[-5:])
        mm.destroy(h)
