"""The FP64 sums' tables (ggem_smooth64.cuh, written by gen_fftab.py fp64): the
smooth parts of the GGEM local kernels as degree-10 pieces in s = 2 alpha^2 r^2.
Truncation is below 2e-17 of the function's largest value, the coefficients and
the Horner steps are rounded to doubles: 5e-16 of that value holds both."""
import pathlib
import re

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
HDR = (pathlib.Path(__file__).resolve().parents[1] / "paper_1109_6587_gb300" / "csrc" /
       "ggem_smooth64.cuh")


@pytest.mark.parametrize("k", [0, 1, 2, 3])
def test_tables_match_mpmath(k):
    txt = HDR.read_text()
    n = int(re.search(r"GGEM_SMOOTH64_NINT (\d+)", txt).group(1))
    deg = int(re.search(r"GGEM_SMOOTH64_DEG (\d+)", txt).group(1))
    num = r"-?0x[0-9a-f.]+p[-+]?\d+"
    v = [float.fromhex(h) for h in re.findall(num, txt[txt.index("kSmooth64[4][%d]" % (deg + 1)):])]
    tab = np.array(v).reshape(4, deg + 1, n)
    mp.mp.dps = 40
    c = mp.sqrt(2 / mp.pi)

    def im(m, s):
        return mp.hyp1f1(mp.mpf(m + 1) / 2, mp.mpf(m + 3) / 2, -s / 2) / (m + 1)
    f = [lambda s: c * (im(0, s) + mp.exp(-s / 2)), lambda s: c * im(2, s),
         lambda s: c * im(4, s) / 3, lambda s: c * mp.exp(-s / 2) / 6][k]
    top = float(f(mp.mpf(0)))
    for s in np.concatenate([np.linspace(0.0, n - 0.6, 200), [0.5, 1.5, 2.4999999]]):
        i = int(round(s))
        p = 0.0
        for d in range(deg, -1, -1):
            p = p * (s - i) + tab[k, d, i]
        assert abs(p - float(f(mp.mpf(float(s))))) < 5e-16 * top
