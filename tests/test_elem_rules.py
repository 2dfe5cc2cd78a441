"""The FP32 element rule's dispatch (ggem_elem32.cu) re-enacted in FP64: what its
point lists per cell, and its binning of triangles by centroid, change in the double
layer's local sums against the 16 points of every triangle within r_cut.

Bounds: the lists below 2e-7 (rms of the differences over the rms sum; two orders of
FP32 summation differ by 2e-7 to 7e-7), the binning below 1e-6 of the largest sum (a
tenth of the mixed path's bar)."""
import pathlib
import re

import numpy as np
import pytest

from oracle import oracle as O
from paper_1109_6587_gb300 import workloads as W

SRC = (pathlib.Path(__file__).resolve().parents[1] / "paper_1109_6587_gb300" / "csrc" /
       "ggem_elem32.cu").read_text()
BOX = W.Box(16.0, 16.0, 6.0, -3.0, 32, 33, 32)


def _const(name):
    return float(re.search(r"\b%s = ([0-9.]+)" % name, SRC).group(1))


def _rules():
    """(barycentric weights [n][3], weights [n]) of the three lists, area 1/2."""
    t, w = O.gauss_legendre01(4)
    p0, w0 = [], []
    for a in range(16):
        eta = t[a >> 2]
        xi = (1 - eta) * t[a & 3]
        p0.append([1 - xi - eta, xi, eta])
        w0.append(w[a & 3] * w[a >> 2] * (1 - eta))
    s = np.sqrt(15.0)
    p1, w1 = [[1 / 3] * 3], [9 / 80]
    for b, v in (((6 + s) / 21, (155 + s) / 2400), ((6 - s) / 21, (155 - s) / 2400)):
        for k in range(3):
            p1.append([1 - 2 * b if v_ == k else b for v_ in range(3)])
            w1.append(v)
    p2 = [[2 / 3 if v_ == k else 1 / 6 for v_ in range(3)] for k in range(3)]
    return [(np.array(p0), np.array(w0)), (np.array(p1), np.array(w1)),
            (np.array(p2), np.full(3, 1 / 6))]


def _edge(s):
    return max(np.linalg.norm(s.x[s.tri[:, i]] - s.x[s.tri[:, (i + 1) % 3]], axis=1).max()
               for i in range(3))


class Sums:
    def __init__(self, s, alpha, rcut, seed=0):
        self.s, self.alpha, self.rcut = s, alpha, rcut
        self.q = np.random.default_rng(seed).standard_normal(s.x.shape)
        a, _, _, self.nrm = O.geometry(s.x, s.tri)
        self.pts = []
        for phi, w in _rules():
            x = np.einsum("pv,tvi->tpi", phi, s.x[s.tri])
            g = np.einsum("p,pv,tvi->tpi", w, phi, self.q[s.tri]) * (2 * a)[:, None, None]
            self.pts.append((x, g))
        self.cen = s.x[s.tri].mean(1)
        n = [int(L / (rcut / 3)) for L in (BOX.Lx, BOX.W, BOX.Lz)]
        self.n, self.h = np.array(n), np.array([BOX.Lx, BOX.W, BOX.Lz]) / n
        self.o = np.array([0.0, BOX.y0, 0.0])

    def terms(self, t, lst, tri=slice(None)):
        """(terms [triangle][point][3], distances) at node t."""
        x, g = (a[tri] for a in self.pts[lst])
        d = self.s.x[t] - x
        for c, L in ((0, BOX.Lx), (2, BOX.Lz)):
            d[..., c] -= L * np.round(d[..., c] / L)
        r = np.linalg.norm(d, axis=-1)
        al, sp, n = self.alpha, np.sqrt(np.pi), self.nrm[t]
        from scipy.special import erfc
        ec, ex = erfc(al * r), np.exp(-(al * r) ** 2)
        xg, xn, gn = (d * g).sum(-1), d @ n, g @ n
        D = -6 * ec / r ** 5 - 12 * al / sp * ex / r ** 4 - 8 * al ** 3 / sp * ex / r ** 2
        E = 4 * al ** 3 / sp * ex
        v = ((D * xg * xn + E * gn)[..., None] * d + (E * xn)[..., None] * g
             + (E * xg)[..., None] * n)
        return v, r

    def cell_distance(self, t):
        """Distance from node t to the box of the cell of each triangle's centroid."""
        c = self.cen - self.o
        for k, L in ((0, BOX.Lx), (2, BOX.Lz)):
            c[:, k] %= L
        ic = np.clip(np.floor(c / self.h), 0, self.n - 1)
        mid = (ic + 0.5) * self.h + self.o
        d = self.s.x[t] - mid
        for k, L in ((0, BOX.Lx), (2, BOX.Lz)):
            d[:, k] -= L * np.round(d[:, k] / L)
        return np.linalg.norm(np.maximum(np.abs(d) - 0.5 * self.h, 0.0), axis=1)


@pytest.mark.parametrize("level,alpha_h", [(3, 0.2), (3, 0.33), (2, 0.33), (3, 0.5), (2, 0.8)])
def test_lists(level, alpha_h):
    """Both lists active up to alpha h = 0.33, list 1 alone beyond."""
    s = W.suspension(6, BOX, level=level, radius=0.93, seed=level)
    h = _edge(s)
    alpha = alpha_h / h
    rcut = 4.0 / alpha
    far1 = _const("kFarEdges") * h
    far2 = max(far1, _const("kDimRadius") / alpha) if alpha_h <= _const("kDimEdge") + 1e-9 else np.inf
    assert far1 < 0.85 * rcut
    S = Sums(s, alpha, rcut)
    diff, ref, used = [], [], set()
    for t in np.random.default_rng(1).choice(len(s.x), 60, replace=False):
        own = (s.tri == t).any(1)
        d = S.cell_distance(t)
        lst = np.where(d >= far2, 2, np.where(d >= far1, 1, 0))
        keep = ~own & (d <= rcut)
        full = S.terms(t, 0, keep)[0].sum((0, 1))
        mix = sum(S.terms(t, k, keep & (lst == k))[0].sum((0, 1)) for k in range(3))
        used |= set(lst[keep])
        diff.append(mix - full)
        ref.append(full)
    assert used == ({0, 1} if far2 == np.inf else {0, 1, 2})
    diff, ref = np.array(diff), np.array(ref)
    rms = np.sqrt((diff ** 2).mean() / (ref ** 2).mean())
    assert rms < 2e-7, rms


@pytest.mark.parametrize("rf,coarse,radius", [(None, 1, 1.1), (None, 2, 1.1), (4.0, 1, 1.3),
                                              (5.0, 1, 1.3), (6.0, 0, 1.3)])
@pytest.mark.parametrize("fine", [1, 3])
def test_centroid_binning_at_its_line(rf, coarse, radius, fine):
    """On both lines (rf None: r_cut = kBinCut / alpha as well).  The longest edge for which triangles are still binned by centroid: points
    within r_cut in cells beyond it are left out, points beyond it in cells within
    are counted; a coarse sphere beside a fine (or another coarse) one."""
    line, rf = _const("kBinRadius"), rf or _const("kBinCut")
    a = W.suspension(1, BOX, level=coarse, radius=radius, centres=np.array([[4.0, 0.1, 5.0]]))
    # alpha (r_cut - 2 h / 3) = line, r_cut = rf / alpha
    alpha = (rf - line) / (2.0 * _edge(a) / 3.0)
    rcut = rf / alpha
    assert 2 * rcut < min(BOX.Lx, BOX.Lz)
    # the second sphere near the first, or (r_cut is long there) across r_cut from it
    b = W.suspension(1, BOX, level=max(fine, coarse), radius=0.9,
                     centres=np.array([[4.0 + max(2.25, rcut), -0.2, 5.2]]))
    s = W.Suspension(BOX, np.concatenate([a.x, b.x]),
                     np.concatenate([a.tri, b.tri + len(a.x)]).astype(np.int32),
                     np.concatenate([a.particle, b.particle + 1]),
                     np.concatenate([a.centres, b.centres]), 1.0)
    S = Sums(s, alpha, rcut)
    worst, top = 0.0, 0.0
    for t in range(0, len(s.x), max(1, len(s.x) // 80)):
        own = (s.tri == t).any(1)
        v, r = S.terms(t, 0, ~own)
        d = S.cell_distance(t)[~own]
        inside = (r < rcut)[..., None]
        strict = (v * inside).sum((0, 1))
        binned = v[d <= rcut].sum((0, 1))
        worst = max(worst, np.abs(binned - strict).max())
        top = max(top, np.abs(strict).max())
    assert worst < 1e-6 * top, worst / top
