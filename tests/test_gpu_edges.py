"""Dispatch edges of the local sums, the interpolation and the element lists, with the
counts taken from the device's multiprocessors: both search reaches, velocity and stress
in one launch with one thread per target, and lists that shrink and grow on one plan.
FP64 1e-10, mixed 1e-5, the paths' bars."""
import numpy as np
import pytest

from _parity import assert_close
from test_gpu_local_split import _direct

from oracle import oracle as O
from paper_1109_6587_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-10, "mixed": 1e-5, "fp64_emulated": 1e-10}


def _nsm():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _points(box, rng, k):
    return rng.uniform(0.0, 1.0, (k, 3)) * [box.Lx, box.W, box.Lz] + [0, box.y0, 0]


@pytest.mark.parametrize("quadrature", ["nodal", "element"])     # search reach 2, 3
@pytest.mark.parametrize("prec,per_sm", [("fp64", 2), ("mixed", 24)])
@pytest.mark.parametrize("more", [0, 1])                         # four warps per target, one
def test_local_sum_split(ggem, quadrature, prec, per_sm, more):
    box = W.Box(16.0, 14.0, 6.0, -3.0, 32, 33, 32)
    n_tgt = per_sm * _nsm() + more
    rng = np.random.default_rng(n_tgt)
    xs, xt, g = _points(box, rng, 777), _points(box, rng, n_tgt), rng.standard_normal((777, 3))
    P = ggem.Plan.for_box(box, alpha=1.0, precision=prec, quadrature=quadrature,
                          max_points=max(1000, n_tgt))
    alpha, rc = P.info()
    ur, sr = _direct(box, alpha, rc, xs, g, xt)
    for wu, ws in ((True, False), (False, True), (True, True)):
        u, s = P.local_sum(xs, g, xt, want_u=wu, want_sigma=ws)
        if wu:
            assert_close(u, ur, TOL[prec])
        if ws:
            assert_close(s, sr, TOL[prec])
    P.check()
    P.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("more", [-1, 0])                        # 8 threads per target, one
def test_velocity_and_stress(ggem, prec, more):
    box = W.Box(16.0, 16.0, 6.0, -3.0, 32, 33, 32)
    n_tgt = 128 * _nsm() + more
    rng = np.random.default_rng(4)
    xs, xt = _points(box, rng, 300), _points(box, rng, n_tgt)
    g = rng.standard_normal((300, 3))
    P = ggem.Plan.for_box(box, precision=prec, max_points=n_tgt)
    u, s = P.point_forces(xs, g, xt, want_u=True, want_sigma=True)
    P.check()
    P.close()
    pick = np.unique(np.concatenate([[0, n_tgt - 1], rng.choice(n_tgt, 200, replace=False)]))
    ur, sr = O.point_forces(box, xs, g, xt=xt[pick], want_sig=True)
    assert_close(u[pick], ur, TOL[prec])
    assert_close(s[pick], np.stack([sr[:, i, j] for i, j in O._SYM6], axis=1), TOL[prec])


@pytest.mark.parametrize("prec", ["mixed", "fp64_emulated"])
def test_lists_grow_and_shrink(ggem, prec):
    """A small mesh, one 12 times larger, the small one again; then large triangles (points
    binned one by one) and the first once more."""
    box = W.Box(16.0, 16.0, 6.0, -3.0, 32, 33, 32)
    small = W.suspension(1, box, level=2, radius=0.9)
    large = W.suspension(3, box, level=3, radius=0.95, seed=2)
    coarse = W.suspension(2, box, level=0, radius=1.9, seed=1)
    P = ggem.Plan.for_box(box, precision=prec, quadrature="element", max_points=len(large.x),
                          max_tris=len(large.tri))
    for s in (small, large, small, coarse, small):
        q = np.random.default_rng(len(s.x)).standard_normal(s.x.shape)
        tg = np.arange(0, len(s.x), max(1, len(s.x) // 100))
        P.mesh_set(s.x, s.tri)
        assert_close(P.single_layer(q)[tg], O.single_layer(s, q, targets=tg), TOL[prec])
        assert_close(P.double_layer(q)[tg], O.double_layer(s, q, targets=tg), TOL[prec])
    P.check()
    P.close()
