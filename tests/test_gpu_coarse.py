"""Mixed element-rule plans on meshes whose triangles are large against r_cut, and with
r_cut below 4 / alpha: every quadrature point within r_cut counts and none beyond it,
against the FP64 oracle (the mixed path's bar, 1e-5)."""
import numpy as np
import pytest

from _parity import assert_close

from oracle import oracle as O
from paper_1109_6587_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL_MIXED = 1e-5


def _layers(ggem, s, q, tg, quadrature, **kw):
    import torch
    P = ggem.Plan.for_box(s.box, precision="mixed", quadrature=quadrature, max_points=len(s.x),
                          max_tris=len(s.tri), **kw)
    alpha, rc = P.info()
    P.mesh_set(s.x, s.tri)
    w = P.single_layer(torch.as_tensor(q, device="cuda")).cpu().numpy()[tg]
    v = P.double_layer(torch.as_tensor(q, device="cuda")).cpu().numpy()[tg]
    P.check()
    P.close()
    ref = dict(quadrature=quadrature, targets=tg, alpha=alpha, rcut=rc)
    return (w, v), (O.single_layer(s, q, **ref), O.double_layer(s, q, **ref))


def _check(ggem, s, tg, **kw):
    q = np.random.default_rng(5).standard_normal(s.x.shape)
    out, ref = _layers(ggem, s, q, tg, "element", **kw)
    for a, b in zip(out, ref):
        assert_close(a, b, TOL_MIXED)


def _beside(level):
    """A fine sphere beside one of radius 2 (longest edge 2.1, 1.2, 0.65, 0.33 r_cut)."""
    box = W.Box(8.0, 8.0, 6.0, -3.0, 64, 65, 64)
    a = W.suspension(1, box, level=3, radius=0.4, centres=np.array([[6.5, 0.1, 4.0]]))
    b = W.suspension(1, box, level=level, radius=2.0, centres=np.array([[4.0, 0.0, 4.0]]))
    n = len(a.x)
    return n, W.Suspension(box, np.concatenate([a.x, b.x]),
                           np.concatenate([a.tri, b.tri + n]).astype(np.int32),
                           np.concatenate([a.particle, b.particle + 1]),
                           np.concatenate([a.centres, b.centres]), 1.0)


@pytest.mark.parametrize("level", [1, 2, 3])
@pytest.mark.parametrize("where", ["fine", "all"])
def test_large_triangles(ggem, level, where):
    n, s = _beside(level)
    tg = np.arange(0, n, 7)
    if where == "all":
        tg = np.concatenate([tg[::3], np.arange(n, len(s.x), 1 + (len(s.x) - n) // 60)])
    _check(ggem, s, tg)


def test_twice_the_cutoff(ggem):
    """The longest edge 2.1 r_cut.  The 12-node sphere's FP32 global part alone is 0.4e-5 to
    1.6e-5 off there, by the density; element and nodal plans share it, so their difference
    shows the local part."""
    n, s = _beside(0)
    tg = np.concatenate([np.arange(0, n, 7), np.arange(n, len(s.x))])
    q = np.random.default_rng(5).standard_normal(s.x.shape)
    eo, er = _layers(ggem, s, q, tg, "element")
    no, nr = _layers(ggem, s, q, tg, "nodal")
    for a, b, c, d in zip(eo, no, er, nr):
        assert np.abs((a - b) - (c - d)).max() < TOL_MIXED * np.abs(c).max()


@pytest.mark.parametrize("n_p", [1, 100])            # four warps per target, one
def test_many_targets(ggem, n_p):
    box = W.Box(32.0, 32.0, 8.0, -4.0, 64, 33, 64)
    s = W.suspension(n_p, box, level=2, radius=1.1, seed=3)
    _check(ggem, s, np.arange(0, len(s.x), max(1, len(s.x) // 150)), alpha=4.0)


@pytest.mark.parametrize("rf", [2.0, 3.0, 3.9])
def test_short_cutoff(ggem, rf):
    s = W.suspension(4, W.Box(16.0, 16.0, 6.0, -3.0, 32, 33, 32), level=2, radius=0.9)
    _check(ggem, s, np.arange(0, len(s.x), 5), rcut_factor=rf)
