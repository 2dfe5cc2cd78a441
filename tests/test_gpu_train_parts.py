"""BF16 training: minibatches whose gradient parts are stored per 128 rows (up to
64 parts) and larger ones that add with atomics give the same steps, also with a
partial last tile; the parted gradient is bitwise reproducible."""
import numpy as np
import pytest

from paper_1109_6587_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ggem():
    from paper_1109_6587_gb300 import _build

    _build.build()
    from paper_1109_6587_gb300 import ggem as G
    return G


def _samples(n):
    rng = np.random.default_rng(n)
    F = rng.standard_normal((n, 12))
    return F, np.tanh(F[:, :3]) + 0.1 * rng.standard_normal((n, 3))


@pytest.mark.parametrize("rows", [1, 127, 129, 2048, 8192, 8193])
def test_one_step(ggem, rows):
    """One Adam step on all rows against the full-batch gradient (atomics) of the
    same model: m1 = 0.1 g, so the first moments must agree with 0.1 g to the
    rounding of FP32 sums (1e-5 of the largest entry of each layer's gradient)."""
    F, T = _samples(rows)
    P = ggem.Plan.for_box(W.box_single_sphere(), precision="mixed", max_points=256, max_tris=256)
    P.mlp_train(F, T, init=True, seed=3, epochs=1, batch=rows, lr=1e-12)
    m = P.mlp_adam_state()[0]
    P2 = ggem.Plan.for_box(W.box_single_sphere(), precision="mixed", max_points=256, max_tris=256)
    P2.mlp_train(F, T, init=True, seed=3, epochs=1, batch=rows, lr=1e-12)
    _, g = P2.mlp_train(F, T, init=False, epochs=0, batch=rows, want_grad=True)
    for a, b in ((0, 1664), (1664, 18176), (18176, 34688), (34688, 35075)):
        assert np.abs(m[a:b] - 0.1 * g[a:b]).max() <= 1e-5 * np.abs(0.1 * g[a:b]).max()
    if rows <= 8192:                    # parts: fixed order of summation
        assert np.array_equal(m, P2.mlp_adam_state()[0])
    P.check()
    P2.check()
