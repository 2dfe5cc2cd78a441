"""The double-float element rule's tables (ggem_fftab.cuh, written by
gen_fftab.py): the smooth parts of the GGEM local kernels as functions of
s = 2 alpha^2 r^2, as degree-9 pieces on |s - i| <= 1/2 in float pairs.  Evaluated
in FP64 from the header they agree with mpmath to 2e-15 of the function's
largest value (the pairs carry 48 bits), and with 1/rho they reproduce the local
kernels of Eq. (local)."""
import math
import pathlib
import re

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
HDR = pathlib.Path(__file__).resolve().parents[1] / "paper_1109_6587_gb300" / "csrc" / "ggem_fftab.cuh"


def _tables():
    txt = HDR.read_text()
    a, b = txt.index("float2 kFFPair"), txt.index("float4 kFFTail")
    num = r"(-?0x[0-9a-f.]+p[-+]?\d+)f"
    pair = [float.fromhex(v) for v in re.findall(num, txt[a:b])]
    tail = [float.fromhex(v) for v in re.findall(num, txt[b:])]
    n = int(re.search(r"GGEM_FF_NINT (\d+)", txt).group(1))
    return np.array(pair).reshape(4, 7, n, 2), np.array(tail).reshape(4, n, 3), n


def _eval(k, s):
    pair, tail, _ = _tables()
    i = int(round(s))
    u, p = s - i, 0.0
    for c in tail[k, i][::-1]:
        p = p * u + c
    for d in range(6, -1, -1):
        p = p * u + pair[k, d, i].sum()
    return p


@pytest.mark.parametrize("k", [0, 1, 2, 3])
def test_tables_match_mpmath(k):
    mp.mp.dps = 40
    c = mp.sqrt(2 / mp.pi)

    def im(m, s):
        return mp.hyp1f1(mp.mpf(m + 1) / 2, mp.mpf(m + 3) / 2, -s / 2) / (m + 1)
    f = [lambda s: c * (im(0, s) + mp.exp(-s / 2)), lambda s: c * im(2, s),
         lambda s: c * im(4, s) / 3, lambda s: c * mp.exp(-s / 2) / 6][k]
    top = float(f(mp.mpf(0)))
    n = _tables()[2]
    for s in np.concatenate([np.linspace(0.0, n - 0.5001, 200), [0.5, 1.5, 2.4999999]]):
        assert abs(_eval(k, s) - float(f(mp.mpf(float(s))))) < 2e-15 * top


@pytest.mark.parametrize("x", [0.3, 1.0, 2.2, 3.7])
def test_tables_give_the_local_kernels(x):
    """x = alpha r (alpha = 1): A, B of G^l and D, E of T^l in closed form."""
    r, lam = x, math.sqrt(2.0)
    rho, s, sp = lam * r, 2.0 * r * r, math.sqrt(math.pi)
    ec, ex = math.erfc(r), math.exp(-r * r)
    A = ec / r - 2 / sp * ex
    B = ec / r ** 3 + 2 / sp * ex / r ** 2
    D = -6 * ec / r ** 5 - 12 / sp * ex / r ** 4 - 8 / sp * ex / r ** 2
    E = 4 / sp * ex
    assert lam * (1 / rho - _eval(0, s)) == pytest.approx(A, rel=0, abs=1e-14 / r)
    assert lam ** 3 * (1 / rho ** 3 - _eval(1, s)) == pytest.approx(B, rel=0, abs=1e-13 / r ** 3)
    assert 6 * lam ** 5 * (_eval(2, s) - rho ** -5) == pytest.approx(D, rel=0, abs=1e-13 / r ** 5)
    assert 6 * lam ** 3 * _eval(3, s) == pytest.approx(E, rel=0, abs=1e-14)
