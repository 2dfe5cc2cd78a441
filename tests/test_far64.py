"""The local kernels as the FP64 sums form them (ggem_smooth64.cuh): near the target
the singular part less a table, farther out a table of the scaled kernel.  Relative to
the kernels themselves both hold 1e-14 up to the tables' end (the difference loses a
factor of up to 12 of the unit rounding's few multiples before the far tables take over;
their truncation is below 1e-15)."""
import math
import pathlib
import re

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
SRC = pathlib.Path(__file__).resolve().parents[1] / "paper_1109_6587_gb300" / "csrc"


def _table(txt, name, funcs, deg, n):
    a = txt.index("%s[%d][%d][%d] = {" % (name, funcs, deg + 1, n))
    v = re.findall(r"-?0x[0-9a-f.]+p[-+]?\d+", txt[a:txt.index("};", a)])
    return np.array([float.fromhex(h) for h in v]).reshape(funcs, deg + 1, n)


def _kernels(s):
    """A, B and -D / 6 of Eq. (local) in units of 1 / (sqrt(2) alpha)."""
    s = mp.mpf(s)
    x, rho = mp.sqrt(s / 2), mp.sqrt(s)
    ec, w = mp.erfc(x), 2 * x * mp.exp(-x * x) / mp.sqrt(mp.pi)
    return (ec - w) / rho, (ec + w) / rho ** 3, (ec + w * (1 + 2 * x * x / 3)) / rho ** 5


@pytest.mark.parametrize("k", [0, 1, 2])
def test_relative_accuracy(k):
    txt = (SRC / "ggem_smooth64.cuh").read_text()
    n = int(re.search(r"GGEM_SMOOTH64_NINT (\d+)", txt).group(1))
    deg = int(re.search(r"GGEM_SMOOTH64_DEG (\d+)", txt).group(1))
    near = _table(txt, "kSmooth64", 4, deg, n)[k]
    far = _table(txt, "kFar64", 3, deg, n)[k]
    line = [int(v) for v in re.search(r"far = i >= \(F == 0 \? (\d+) : (\d+)\)",
                                      (SRC / "ggem_local.cu").read_text()).groups()]
    i0 = line[0] if k < 2 else line[1]
    mp.mp.dps = 40
    for s in np.concatenate([np.linspace(2.0, n - 0.6, 400), [i0 - 0.5000001, i0 - 0.4999999]]):
        s = float(s)
        i, ir = int(round(s)), 1.0 / math.sqrt(s)
        p = 0.0
        for c in (far if i >= i0 else near)[::-1, i]:
            p = p * (s - i) + c
        ref = _kernels(s)[k]
        f = ir ** (2 * k + 1) * p if i >= i0 else ir ** (2 * k + 1) - p
        assert abs(float(f / ref) - 1) < 1e-14, s
