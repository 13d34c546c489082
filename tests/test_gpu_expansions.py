"""The truncated expansions themselves: the deflection at every dealing of
the order against the same sums (P2M, M2L, P2L, L2L, re-centring; App. C.2)
in FP64 on the host, cut at the same order, so that a wrong or missing row
shows whatever the truncation leaves out."""
import math

import numpy as np
import pytest

import paper_2506_02114_gb300 as mm
import synthetic
from _metrics import DEFLECTION_TOL, deflection_rel_error

pytestmark = pytest.mark.gpu

DEEPEST = 21     # levels of the tree below the root
NEAR = 5         # sub-cells a side of the block whose stars are summed directly


class HostExpansions:
    """Locals of the tree of stars (m, z), root [-R0, R0]^2, order p, about
    every node asked for.  The multipole of a node is formed from its stars:
    shifting truncated multipoles to a parent is exact below the cut."""

    def __init__(self, m, pos, R0, limit, p):
        self.m, self.z, self.R0, self.limit, self.p = m, pos[:, 0] + 1j * pos[:, 1], R0, limit, p
        self.cell = np.clip(np.floor((pos + R0) * ((1 << DEEPEST) / (2.0 * R0))), 0,
                            (1 << DEEPEST) - 1).astype(np.int64)
        self.stars, self.loc, self.mult = {}, {}, {}
        self.k = np.arange(1, p + 1)
        self.binom = np.array([[float(math.comb(l + k - 1, k - 1)) for k in self.k] for l in self.k])

    def inside(self, level, x, y):
        """Indices of the stars in a cell."""
        key = (level, x, y)
        if key not in self.stars:
            if level == 0:
                i = np.arange(len(self.m))
            else:
                i = self.inside(level - 1, x >> 1, y >> 1)
                i = i[((self.cell[i] >> (DEEPEST - level)) == (x, y)).all(1)]
            self.stars[key] = i
        return self.stars[key]

    def around(self, level, x, y):
        side = 1 << level
        return [(x + dx, y + dy) for dy in (-1, 0, 1) for dx in (-1, 0, 1)
                if 0 <= x + dx < side and 0 <= y + dy < side]

    def split(self, level, x, y):
        return level < DEEPEST and sum(len(self.inside(level, *c))
                                       for c in self.around(level, x, y)) > self.limit

    def is_node(self, level, x, y):
        return level == 0 or (self.split(level - 1, x >> 1, y >> 1)
                              and self.is_node(level - 1, x >> 1, y >> 1))

    def centre(self, level, x, y):
        L = self.R0 / (1 << level)
        return complex(-self.R0 + (2 * x + 1) * L, -self.R0 + (2 * y + 1) * L), L

    def multipole(self, level, x, y):
        key = (level, x, y)
        if key not in self.mult:
            zc, L = self.centre(*key)
            i = self.inside(*key)
            zeta = ((self.z[i] - zc) / L)[:, None] ** self.k
            self.mult[key] = (self.m[i].sum(), -(self.m[i][:, None] * zeta).sum(0) / self.k)
        return self.mult[key]

    def local(self, level, x, y):
        """c_1 .. c_p of a node."""
        key = (level, x, y)
        if level < 2:
            return np.zeros(self.p, complex)
        if key not in self.loc:
            zc, L = self.centre(*key)
            up = self.local(level - 1, x >> 1, y >> 1)
            c = recentre(up, complex(0.5 if x & 1 else -0.5, 0.5 if y & 1 else -0.5), 0.5, self.p)
            for qx, qy in self.around(level - 1, x >> 1, y >> 1):
                if (qx, qy) == (x >> 1, y >> 1):
                    continue
                if self.split(level - 1, qx, qy):
                    for cx, cy in [(2 * qx + i, 2 * qy + j) for i in (0, 1) for j in (0, 1)]:
                        if max(abs(cx - x), abs(cy - y)) > 1:
                            a0, a = self.multipole(level, cx, cy)
                            iz = 1.0 / (2.0 * complex(cx - x, cy - y))
                            c += iz ** self.k * (self.binom @ (a * (-iz) ** self.k) - a0 / self.k)
                elif max(abs(2 * qx + 0.5 - x), abs(2 * qy + 0.5 - y)) > 2.0:
                    i = self.inside(level - 1, qx, qy)
                    w = (self.z[i] - zc) / L
                    c -= (self.m[i][:, None] / (self.k * w[:, None] ** self.k)).sum(0)
            self.loc[key] = c
        return self.loc[key]

    def leaf(self, cx, cy):
        level = 0
        while self.split(level, cx >> (DEEPEST - level), cy >> (DEEPEST - level)):
            level += 1
        return level, cx >> (DEEPEST - level), cy >> (DEEPEST - level)

    def near(self, level, x, y):
        """Stars of the leaf's neighbourhood: same-level cells that are nodes,
        else the coarser leaf over them, once."""
        cells = set()
        for q in self.around(level, x, y):
            cells.add((level,) + q if self.is_node(level, *q) else (level - 1, q[0] >> 1, q[1] >> 1))
        return np.concatenate([self.inside(*c) for c in sorted(cells)])

    def slope(self, z, sub, terms):
        """dpsi/dz at z: the sub-cell's expansion cut at `terms`, and its direct stars."""
        c = np.clip(np.floor((np.array([z.real, z.imag]) + self.R0)
                             * ((1 << DEEPEST) / (2.0 * self.R0))), 0, (1 << DEEPEST) - 1).astype(int)
        level, x, y = self.leaf(int(c[0]), int(c[1]))
        zc, L = self.centre(level, x, y)
        sh = DEEPEST - level - sub
        zq, Lq = self.centre(level + sub, int(c[0]) >> sh, int(c[1]) >> sh)
        d = recentre(self.local(level, x, y), (zq - zc) / L, Lq / L, terms)
        i = self.near(level, x, y)
        off = self.z[i] - zq
        far = (np.maximum(abs(off.real), abs(off.imag)) >= NEAR * Lq) if sub else np.zeros(len(i), bool)
        n = np.arange(1, terms + 1)
        w = off[far] / Lq
        d = d - (self.m[i[far]][:, None] / (n * w[:, None] ** n)).sum(0)
        return ((n * d * ((z - zq) / Lq) ** (n - 1)).sum() / Lq
                + (self.m[i[~far]] / (z - self.z[i[~far]])).sum())


def recentre(c, u, r, terms):
    """sum_l c_l zeta^l about u, in units of r: the first `terms` coefficients."""
    p = len(c)
    return np.array([r ** n * sum(math.comb(l, n) * c[l - 1] * u ** (l - n) for l in range(n, p + 1))
                     for n in range(1, min(terms, p) + 1)], complex)


@pytest.mark.parametrize("p", [1, 2, 3, 5, 20, 31, 32, 33, 40, 43, 63, 64])
@pytest.mark.parametrize("leaf", [4, 100])
@pytest.mark.parametrize("sub", [-1, 1, 2])
def test_deflection_is_that_of_the_cut_expansions(p, leaf, sub):
    m, pos = synthetic.star_field(17, 700, 30.0, synthetic.SALPETER_01_1)
    kappa, gamma, s = 0.4, 0.3, 0.2
    h = mm.create(kappa, gamma, s, m, pos, 1.0, 16, fmm_order=p, leaf_size=leaf, sub_levels=sub,
                  img_half=(6.0, 6.0), ray_grid=(241, 241))
    z = 12.0 * np.stack([synthetic.uniform(8, 0, 150), synthetic.uniform(8, 1, 150)], 1) - 6.0
    w = mm.shoot_points(h, z)
    st = mm.get_stats(h)
    mm.destroy(h)
    host = HostExpansions(m, pos, st["root_half_length"], leaf, p)
    par = type("P", (), dict(kappa=kappa, gamma=gamma, kappa_star=(1 - s) * kappa))
    slope = np.array([host.slope(complex(*q), st["sub_levels"], st["eval_order"]) for q in z])
    macro = np.stack([(1 - kappa + gamma) * z[:, 0], (1 - kappa - gamma) * z[:, 1]], 1)
    w_host = macro - np.stack([slope.real, -slope.imag], 1) + par.kappa_star * z
    err = deflection_rel_error(par, z, w, w_host).max()
    assert err <= DEFLECTION_TOL, err
