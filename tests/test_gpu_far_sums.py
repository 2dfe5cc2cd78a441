"""FP64 local sums at targets whose sources are all far away: the returned values have
their digits, also for a cutoff beyond the tables' end (6.02 / alpha), and no term
within r_cut is left out.  Relative to the largest component: the kernels fall by
2 alpha r per unit of alpha r, so positions good to a few 1e-15 of the box give 4e-14
at most; bar 1e-13.  (Velocity and stress in one call take erfc's own route, 1e-13 up
to 4 / alpha.)"""
import math

import numpy as np
import pytest

from paper_1109_6587_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-13


def _pair(alpha, d, g):
    r = math.sqrt(float(d @ d))
    x, sp, xg = alpha * r, math.sqrt(math.pi), float(d @ g)
    ec, ex = math.erfc(x), math.exp(-x * x)
    u = (ec / r - 2 * alpha / sp * ex) * g + (ec / r ** 3 + 2 * alpha / sp * ex / r ** 2) * xg * d
    D = (-6 * ec / r ** 5 - 12 * alpha / sp * ex / r ** 4 - 8 * alpha ** 3 / sp * ex / r ** 2) * xg
    E = 4 * alpha ** 3 / sp * ex
    s = [D * d[i] * d[j] + E * (g[i] * d[j] + g[j] * d[i] + (xg if i == j else 0.0))
         for i, j in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))]
    return u / (8 * math.pi), np.array(s) / (8 * math.pi)


@pytest.mark.parametrize("quadrature", ["nodal", "element"])     # both search reaches
@pytest.mark.parametrize("rf,ar", [(4.0, 1.3), (4.0, 1.6), (4.0, 1.7), (4.0, 2.9), (4.0, 3.95),
                                   (6.5, 5.0), (6.5, 5.95), (6.5, 6.01), (6.5, 6.03),
                                   (6.5, 6.45), (7.9, 7.8)])
def test_far_pair(ggem, quadrature, rf, ar):
    box = W.Box(16.0, 16.0, 6.0, -3.0, 32, 33, 32)
    rng = np.random.default_rng(int(100 * ar))
    xs = np.array([[8.0, 0.1, 7.0]])
    xt = xs + ar * np.array([[0.8, 0.0, 0.6]])
    g = rng.standard_normal((1, 3))
    P = ggem.Plan.for_box(box, alpha=1.0, rcut_factor=rf, precision="fp64", quadrature=quadrature,
                          max_points=4096)
    ur, sr = _pair(1.0, (xt - xs)[0], g[0])
    for n_tgt in (1, 700):                                       # four warps per target, one
        t = np.repeat(xt, n_tgt, 0)
        u, _ = P.local_sum(xs, g, t, want_u=True)
        _, s = P.local_sum(xs, g, t, want_u=False, want_sigma=True)
        for a, b in ((u, ur), (s, sr)):
            assert np.abs(a - b).max() < TOL * np.abs(b).max()
    if rf == 4.0:
        u, s = P.local_sum(xs, g, xt, want_u=True, want_sigma=True)
        for a, b in ((u, ur), (s, sr)):
            assert np.abs(a - b).max() < TOL * np.abs(b).max()
    P.close()

