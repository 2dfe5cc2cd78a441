"""Double-float element rule against the native FP64 plan (bar 1e-10, the FP64
paths' parity with the oracle): cutoffs inside, at and beyond its tables, open
meshes with ragged cells, the smallest cells and nearly empty neighbour lists."""
import numpy as np
import pytest

from _parity import assert_close

from paper_1109_6587_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL_FP64 = 1e-10


@pytest.fixture(scope="module")
def ggem():
    from paper_1109_6587_gb300 import _build

    _build.build()
    from paper_1109_6587_gb300 import ggem as G
    return G


@pytest.mark.parametrize("rcut_factor", [2.0, 4.0, 6.5])
@pytest.mark.parametrize("mesh", ["sphere", "ragged", "touching"])
def test_matches_fp64_plan(ggem, mesh, rcut_factor):
    box = W.Box(16.0, 12.0, 6.0, -3.0, 32, 33, 32)
    if mesh == "touching":              # surfaces 1e-4 apart: displacements near the grid's step
        s = W.suspension(2, box, level=1, radius=0.9,
                         centres=np.array([[4.0, 0.1, 5.0], [5.8001, 0.1, 5.0]]))
    else:
        s = W.suspension(2, box, level=2, radius=0.93)
    tri = s.tri
    if mesh == "ragged":
        keep = np.random.default_rng(2).permutation(len(tri))[:len(tri) - 53]
        tri = np.ascontiguousarray(tri[np.sort(keep)])
    q = np.random.default_rng(3).standard_normal(s.x.shape)
    used = np.unique(tri)
    out = {}
    for prec in ("fp64", "fp64_emulated"):
        P = ggem.Plan.for_box(box, precision=prec, quadrature="element", max_points=len(s.x),
                              max_tris=len(tri), alpha=1.5, rcut_factor=rcut_factor)
        P.mesh_set(s.x, tri)
        out[prec] = [P.single_layer(q)[used], P.double_layer(q)[used]]
        P.close()
    for a, b in zip(out["fp64_emulated"], out["fp64"]):
        assert_close(a, b, TOL_FP64)
