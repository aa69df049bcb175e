"""The cooling terms that the kernels leave out as too small (kCoolCut and
kCoolExp of csrc/rates.cuh) on the CPU, with the rate functions as the kernels
hold them: a term is left out where its function, times 2^kCoolExp, is below
2^kCoolCut.  Together they must stay below 2^-48 (the accuracy of the float pairs
that hold the sums) of the cooling at every temperature from 10 K to 1e9 K, for
x_HII from its floor 1e-6 to 1 and helium from neutral to ionised."""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_1304_7126_gb300", "csrc", "rates.cuh")


@pytest.mark.parametrize("case_b", [True, False])
def test_left_out_cooling_terms(case_b):
    from paper_1304_7126_gb300 import rt as R
    text = open(HEADER).read()
    cut, scale = (int(re.search(r"constexpr int %s = (-?\d+);" % k, text).group(1)) for k in ("kCoolCut", "kCoolExp"))
    tab = R.rate_functions(case_b)[:11]
    T = np.geomspace(10.0, 1e9, 4001)[:, None]
    Cc, c0, c1, c2, c3, c4, c5 = tab.T
    lnT = np.log(T)
    f = Cc * np.exp(c0 + c1 * lnT + c2 / T - c3 * np.logaddexp(0.0, c4 * lnT + c5))     # [T][term]
    # a value y 2^m is left out by m, with y in [0.99, 4.1)
    out = f * 2.0 ** scale < 4.1 * 2.0 ** cut
    worst = 0.0
    for x in (1e-6, 1e-4, 1e-2, 0.5, 1.0):
        for y2, y3 in ((0.0, 0.0), (1e-6, 0.0), (0.5, 0.1), (0.0, 1.0)):
            he = 0.24 / (4 * 0.76)
            n = {"HI": 1 - x, "HII": x, "HeI": he * (1 - y2 - y3), "HeII": he * y2, "HeIII": he * y3}
            n["ff"] = n["HII"] + n["HeII"] + 4 * n["HeIII"]
            of = [n[k] for k in ("HI", "HI", "HII", "ff", "HeI", "HeII", "HeII", "HeII", "HeII", "HeII", "HeIII")]
            term = f * np.array(of)
            worst = max(worst, float(((term * out).sum(1) / term.sum(1)).max()))
    assert worst < 2.0 ** -48, worst
