"""Local sums: one and four warps per target (the target counts around both rules'
lines), both search reaches, the FP64 tables and their end (r_cut = 6.3 / alpha
lies beyond them), against a direct FP64 sum of Eq. (local) with erfc.
FP64 1e-10, mixed 1e-5, the paths' bars."""
import math

import numpy as np
import pytest

from _parity import assert_close

from paper_1109_6587_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-10, "mixed": 1e-5}


@pytest.fixture(scope="module")
def ggem():
    from paper_1109_6587_gb300 import _build

    _build.build()
    from paper_1109_6587_gb300 import ggem as G
    return G


def _direct(box, alpha, rc, xs, g, xt):
    import torch
    z, x, f = (torch.as_tensor(a, device="cuda") for a in (xt, xs, g))
    d = z[:, None] - x[None]
    for c, L in ((0, box.Lx), (2, box.Lz)):
        d[..., c] -= L * torch.round(d[..., c] / L)
    r = d.norm(dim=-1)
    ec, ex = torch.erfc(alpha * r), torch.exp(-(alpha * r) ** 2)
    sp, xg = math.sqrt(math.pi), (d * f).sum(-1)
    m = (r < rc).to(torch.float64)
    A = m * (ec / r - 2 * alpha / sp * ex)
    B = m * (ec / r ** 3 + 2 * alpha / sp * ex / r ** 2) * xg
    D = m * (-6 * ec / r ** 5 - 12 * alpha / sp * ex / r ** 4
             - 8 * alpha ** 3 / sp * ex / r ** 2) * xg
    E = m * 4 * alpha ** 3 / sp * ex
    u = (A[..., None] * f + B[..., None] * d).sum(1) / (8 * math.pi)
    s = [(D * d[..., i] * d[..., j]
          + E * (f[:, i] * d[..., j] + f[:, j] * d[..., i] + (xg if i == j else 0))).sum(1)
         for i, j in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))]
    return u.cpu().numpy(), (torch.stack(s, 1) / (8 * math.pi)).cpu().numpy()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n_tgt", [1, 304, 305, 3648, 3649])
@pytest.mark.parametrize("rf", [4.0, 6.3])
def test_local_sum(ggem, prec, n_tgt, rf):
    box = W.Box(16.0, 14.0, 6.0, -3.0, 32, 33, 32)
    rng = np.random.default_rng(n_tgt)

    def pts(k):
        return rng.uniform(0.0, 1.0, (k, 3)) * [box.Lx, box.W, box.Lz] + [0, box.y0, 0]
    xs, xt, g = pts(777), pts(n_tgt), rng.standard_normal((777, 3))
    P = ggem.Plan.for_box(box, alpha=1.0, rcut_factor=rf, precision=prec, max_points=4096)
    alpha, rc = P.info()
    ur, sr = _direct(box, alpha, rc, xs, g, xt)
    u, s = P.local_sum(xs, g, xt, want_u=True, want_sigma=True)
    assert_close(u, ur, TOL[prec])
    assert_close(s, sr, TOL[prec])
    u, _ = P.local_sum(xs, g, xt, want_u=True)               # one kind at a time: FP64 tables
    assert_close(u, ur, TOL[prec])
    _, s = P.local_sum(xs, g, xt, want_u=False, want_sigma=True)
    assert_close(s, sr, TOL[prec])
    P.check()
    P.close()
