"""The FP64 block-moment kernel's cos / sin polynomials, read from the kernel source: they are
the fit of csrc/fit_sincos.py, and in 50 digits they stay within the errors that the source
states, up to the phases the kernel uses them for."""
import os
import re
import sys
from decimal import Decimal, localcontext

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1003_1140_gb300", "csrc")
sys.path.insert(0, CSRC)


def _source():
    src = open(os.path.join(CSRC, "rad_accum64.cu")).read()
    table = re.search(r"g_coef64\[3\]\[kMaxP\] = \{(.*?)\};", src, re.S).group(1)
    rows = [[float(v) for v in r.split(",")] for r in re.findall(r"\{([^{}]*)\}", table)]
    lim = re.search(r"kX0 = ([0-9.]+)f, kX1 = ([0-9.]+)f, kX2 = ([0-9.]+)f", src).groups()
    return rows, [float(v) for v in lim]


@pytest.mark.parametrize("row,terms,bound", [(0, 12, 7.8e-17), (1, 16, 2.9e-17), (2, 20, 7.2e-17)])
def test_fp64_moment_polynomials(row, terms, bound):
    import fit_sincos as f
    rows, lim = _source()
    c, x0 = rows[row], lim[row]
    assert len(c) == 20 and not any(c[terms:])
    with localcontext() as ctx:
        ctx.prec = 50
        d = [Decimal(v) for v in c]
        worst = Decimal(0)
        for i in range(1001):
            t = Decimal(x0) * i / 1000
            z, p = -t * t, [Decimal(0), Decimal(0)]
            for j in reversed(range(terms // 2)):
                p = [p[0] * z + d[2 * j], p[1] * z + d[2 * j + 1]]
            cs = f.dec_cos_sin(t)
            worst = max(worst, abs(p[0] - cs[0]), abs(t * p[1] - cs[1]))
    assert 0.9 * bound < worst <= bound
    np.testing.assert_allclose(c[:terms], f.fit_moment64(x0, terms // 2), rtol=1e-4)
