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
    row = re.search(r"g_moment_coef\[kMaxP\] = \{(.*?)\};", src, re.S).group(1)
    x0 = float(re.search(r"kX12 = ([0-9.]+)f", src).group(1))
    return np.array([float(v.strip().rstrip("f")) for v in row.split(",")]), x0


@pytest.mark.parametrize("terms", [12])
def test_moment_polynomials(terms):
    sys.path.insert(0, CSRC)
    import fit_sincos as f
    c, x0 = _source()
    assert len(c) == terms
    t = np.linspace(-x0, x0, 200001)
    z = -t * t
    cos = sum(c[2 * j] * z ** j for j in range(terms // 2))
    sin = t * sum(c[2 * j + 1] * z ** j for j in range(terms // 2))
    assert np.abs(cos - np.cos(t)).max() < 7e-8
    assert np.abs(sin - np.sin(t)).max() < 7e-8
    fit, err = f.fit_moment(x0, terms // 2)
    assert err < 7e-8
    np.testing.assert_allclose(c, fit, rtol=2e-5)
