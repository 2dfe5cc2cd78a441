"""FP32 element rule: point lists per quadrature rule of the triangles, at the
sizes where the lists and cells have their edges, against the FP64 oracle
(the mixed path's bar, 1e-5)."""
import numpy as np
import pytest

from _parity import assert_close

from oracle import oracle as O
from paper_1109_6587_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL_MIXED = 1e-5


@pytest.fixture(scope="module")
def ggem():
    from paper_1109_6587_gb300 import _build

    _build.build()
    from paper_1109_6587_gb300 import ggem as G
    return G


def _mesh(name):
    if name == "one_triangle":          # a single triangle: one step, dummies in 48 of 64 slots
        s = W.suspension(1, W.Box(16.0, 16.0, 6.0, -3.0, 32, 33, 32), level=2, radius=0.97)
        return W.Suspension(s.box, s.x, s.tri[:1], s.particle, s.centres, s.radius)
    if name == "ragged":                # an open mesh, triangle counts not multiples of 4
        s = W.suspension(2, W.Box(16.0, 12.0, 6.0, -3.0, 32, 33, 32), level=2, radius=0.93)
        keep = np.random.default_rng(1).permutation(len(s.tri))[:len(s.tri) - 37]
        return W.Suspension(s.box, s.x, np.ascontiguousarray(s.tri[np.sort(keep)]), s.particle,
                            s.centres, s.radius)
    if name == "two_sizes":             # a fine sphere beside a coarse one: the longest edge rules
        box = W.Box(16.0, 16.0, 6.0, -3.0, 32, 33, 32)
        a = W.suspension(1, box, level=3, radius=0.9, centres=np.array([[4.0, 0.1, 5.0]]))
        b = W.suspension(1, box, level=1, radius=1.1, centres=np.array([[6.3, -0.2, 5.4]]))
        n = len(a.x)
        return W.Suspension(box, np.concatenate([a.x, b.x]),
                            np.concatenate([a.tri, b.tri + n]).astype(np.int32),
                            np.concatenate([a.particle, b.particle + 1]),
                            np.concatenate([a.centres, b.centres]), 1.0)
    lv = {"coarse": 1, "level2": 2, "level3": 3}[name]
    # coarse: 4 edges are beyond 0.85 r_cut (only the 16-point list); level3: mostly the far one
    return W.suspension(2, W.Box(16.0, 16.0, 6.0, -3.0, 32, 33, 32), level=lv, radius=0.94)


@pytest.mark.parametrize("name", ["one_triangle", "ragged", "two_sizes", "coarse", "level2",
                                  "level3"])
def test_lists_match_oracle(ggem, name):
    import torch
    s = _mesh(name)
    n = len(s.x)
    q = np.random.default_rng(5).standard_normal((n, 3))
    P = ggem.Plan.for_box(s.box, precision="mixed", quadrature="element", max_points=n,
                          max_tris=len(s.tri))
    P.mesh_set(s.x, s.tri)
    tg = np.unique(s.tri)[::max(1, len(np.unique(s.tri)) // 150)]
    w = P.single_layer(torch.as_tensor(q, device="cuda")).cpu().numpy()[tg]
    v = P.double_layer(torch.as_tensor(q, device="cuda")).cpu().numpy()[tg]
    P.check()
    P.close()
    with np.errstate(invalid="ignore", divide="ignore"):    # nodes without a triangle
        assert_close(w, O.single_layer(s, q, quadrature="element", targets=tg), TOL_MIXED)
        # (alone, a flat triangle's double layer is its polar rule at nodes of its own plane,
        # a cancelling sum that these lists have no part in)
        if name != "one_triangle":
            assert_close(v, O.double_layer(s, q, quadrature="element", targets=tg), TOL_MIXED)


@pytest.mark.parametrize("alpha_h", [0.32, 0.34])
def test_dim_list_matches_oracle(ggem, alpha_h):
    """The 3-point list on both sides of its rule (alpha times the longest edge
    0.33), with most of the pairs beyond 3 / alpha."""
    import torch
    box = W.Box(16.0, 16.0, 6.0, -3.0, 32, 33, 32)
    s = W.suspension(4, box, level=2, radius=0.9)
    edge = max(np.linalg.norm(s.x[s.tri[:, i]] - s.x[s.tri[:, (i + 1) % 3]], axis=1).max()
               for i in range(3))
    alpha = alpha_h / edge
    q = np.random.default_rng(6).standard_normal(s.x.shape)
    P = ggem.Plan.for_box(box, alpha=alpha, precision="mixed", quadrature="element",
                          max_points=len(s.x), max_tris=len(s.tri))
    P.mesh_set(s.x, s.tri)
    tg = np.arange(0, len(s.x), 5)
    w = P.single_layer(torch.as_tensor(q, device="cuda")).cpu().numpy()[tg]
    v = P.double_layer(torch.as_tensor(q, device="cuda")).cpu().numpy()[tg]
    P.check()
    P.close()
    kw = dict(quadrature="element", targets=tg, alpha=alpha)
    assert_close(w, O.single_layer(s, q, **kw), TOL_MIXED)
    assert_close(v, O.double_layer(s, q, **kw), TOL_MIXED)
