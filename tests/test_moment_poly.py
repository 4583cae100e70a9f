"""The block-moment kernel's cos / sin polynomials, read from the kernel source: they are
the fit of csrc/fit_sincos.py and stay within 7e-8 of cos and sin up to the phase the
kernel uses them for."""
import os
import re
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1003_1140_gb300", "csrc")


def _source():
    src = open(os.path.join(CSRC, "rad_accum32_moment.cu")).read()
    rows = re.search(r"g_moment_coef\[2\]\[kMaxP\] = \{\s*\{(.*?)\},\s*\{(.*?)\}\};", src, re.S)
    lim = [float(v) for v in re.search(r"kX8 = ([0-9.]+)f, kX12 = ([0-9.]+)f", src).groups()]
    return [np.array([float(v.strip().rstrip("f")) for v in r.split(",")]) for r in rows.groups()], lim


@pytest.mark.parametrize("row,terms", [(0, 8), (1, 12)])
def test_moment_polynomials(row, terms):
    sys.path.insert(0, CSRC)
    import fit_sincos as f
    tables, lim = _source()
    c, x0 = tables[row], lim[row]
    assert np.all(c[terms:] == 0.0)
    t = np.linspace(-x0, x0, 200001)
    z = -t * t
    cos = sum(c[2 * j] * z ** j for j in range(terms // 2))
    sin = t * sum(c[2 * j + 1] * z ** j for j in range(terms // 2))
    assert np.abs(cos - np.cos(t)).max() < 7e-8
    assert np.abs(sin - np.sin(t)).max() < 7e-8
    fit, err = f.fit_moment(x0, terms // 2)
    assert err < 7e-8
    np.testing.assert_allclose(c[:terms], fit, rtol=2e-5)
