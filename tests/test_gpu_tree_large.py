"""Trees of many stars: the levels' nodes and the active leaves numbered from
running sums of their groups' counts."""
import math

import numpy as np
import pytest

import paper_2506_02114_gb300 as mm
import synthetic
from _metrics import DEFLECTION_TOL, deflection_rel_error

pytestmark = pytest.mark.gpu


def host_counts(pos, R0, limit):
    """(nodes per level, leaves) of the tree: a node splits when the stars in its
    3 x 3 block of same-level cells exceed the limit, down to level 21."""
    cell = np.clip(np.floor((pos + R0) * ((1 << 21) / (2.0 * R0))), 0, (1 << 21) - 1).astype(np.int64)
    nodes, counts, leaves = np.zeros((1, 2), np.int64), [], 0
    for level in range(22):
        counts.append(len(nodes))
        keys, n = np.unique((cell[:, 0] >> (21 - level) << 32) | (cell[:, 1] >> (21 - level)),
                            return_counts=True)
        block = np.zeros(len(nodes), np.int64)
        for dx in (-1, 0, 1):
            for dy in (-1, 0, 1):
                x, y = nodes[:, 0] + dx, nodes[:, 1] + dy
                k = np.searchsorted(keys, (x << 32) | y).clip(0, len(keys) - 1)
                block += np.where((x >= 0) & (y >= 0) & (keys[k] == ((x << 32) | y)), n[k], 0)
        split = (block > limit) & (level < 21)
        leaves += int((~split).sum())
        nodes = np.concatenate([2 * nodes[split] + (i, j) for i in (0, 1) for j in (0, 1)])
        if not len(nodes):
            break
    return counts, leaves


# nodes of a level, and nodes in all, beyond which running sums number them
# (MM_SUM_GROUPS groups of MM_SPLIT_GROUP and of MM_ACTIVE_GROUP)
LEVEL_SUMS, NODE_SUMS = 8192 * 32, 8192 * 256


@pytest.mark.parametrize("n,limit,level_sums,node_sums", [
    (40000, 3, False, False), (150000, 3, True, False), (400001, 3, True, True)])
def test_levels_of_many_nodes(oracle_mod, n, limit, level_sums, node_sums):
    """Levels whose nodes are numbered from running sums of their groups (a
    partly filled last round of them among these) and from counts added up."""
    u = synthetic.uniform
    R = math.sqrt(n / 3.0)
    pos = 2.0 * R * np.stack([u(31, 0, n), u(31, 1, n)], 1) - R
    m = np.ones(n)
    kappa, gamma, s, p = 0.4, 0.3, 0.0, 20
    grid = dict(img_half=(0.4 * R, 0.4 * R), ray_grid=(301, 301))
    h = mm.create(kappa, gamma, s, m, pos, 1.0, 16, fmm_order=p, leaf_size=limit, **grid)
    st = mm.get_stats(h)
    counts, leaves = host_counts(pos, st["root_half_length"], limit)
    assert (max(counts) > LEVEL_SUMS, sum(counts) > NODE_SUMS) == (level_sums, node_sums)
    for _ in range(2):   # the plan's tree, then the run's
        st = mm.get_stats(h)
        assert (st["nodes"], st["leaves"], st["depth"]) == (sum(counts), leaves, len(counts) - 1)
        assert st["error_bits"] == 0
        z = 0.78 * R * np.stack([u(32, 0, 400), u(32, 1, 400)], 1) - 0.39 * R
        w = mm.shoot_points(h, z)
        par = oracle_mod.derive_params(kappa, gamma, s, m, 1.0, 16, **grid)
        r = math.sqrt(2.0) / (4.0 - math.sqrt(2.0))
        err = deflection_rel_error(par, z, w, oracle_mod.deflect(par, m, pos, z)).max()
        assert err <= DEFLECTION_TOL + 2.2 * (p + 1) * r ** p, err
        mm.run(h, 0)
        mm.run(h, 0)
    mm.destroy(h)
