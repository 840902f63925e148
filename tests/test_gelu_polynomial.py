"""The polynomial behind the CUDA GELU, max(z, 0) - a 2^q(-a) with a = |z|, on the
host: its error with the kernels' fp32 evaluation order, what makes the value
exactly max(z, 0) from Z on, and that the header holds these coefficients (two
other tests, written for a rational function, ask for an error below 2e-6 and
for a denominator, which it has not)."""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def gen():
    pytest.importorskip("scipy")
    from paper_2609_09020_gb300 import gen_gelu
    return gen_gelu, gen_gelu.fit()


def test_error_bound(gen):
    # 5.2e-7 over [-12, 12], most of it the rounding of results near 8
    g, coeffs = gen
    assert g.max_error(coeffs) <= 5.6e-7
    z = np.linspace(-6, 6, 600001)
    from scipy.special import erf
    ref = 0.5 * z * (1 + erf(z / np.sqrt(2)))
    assert np.max(np.abs(g.gelu_fp32(z, coeffs).astype(np.float64) - ref)) <= 5.6e-7


def test_subtracted_part_vanishes_at_the_end_of_the_range(gen):
    # the power at -Z, with two ulps of ex2.approx, stays below EPS, and both are
    # too small to show before that
    g, (c, eps) = gen
    power = 2.0 ** np.polyval([float(np.float32(k)) for k in c[::-1]], -np.float32(g.Z))
    assert power * (1 + 2.0 ** -22) < np.float32(eps) < 3.5e-9


def test_header_constants(gen):
    g, (c, eps) = gen
    text = open(os.path.join(ROOT, "paper_2609_09020_gb300", "csrc", "pic_gelu.cuh")).read()
    values = [np.float32(v) for v in re.findall(r"^\s+(-?[0-9.e+-]+)f,$", text, re.M)]
    assert values == [np.float32(k) for k in c[::-1]] and len(values) == g.DEG + 1
    assert np.float32(re.search(r"kGeluEps = ([0-9.e+-]+)f", text).group(1)) == np.float32(eps)
