"""The polynomials that stand for the stresses at moderate strain, read from the
kernels' header: y(m) = 1 - (1 + m)^-1/2 and q(m) = log(1 + m) / (2 (1 + m)), each
m times a polynomial with FP32 coefficients, over every eigenvalue that the rule
of their use admits (|M| <= kSmallStrain bounds each). The header states a
relative error below 1.5e-8."""
import os
import re

import numpy as np
import pytest

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                      "paper_2503_05046_gb300", "csrc", "common.cuh")


def coefficients(name):
    with open(HEADER) as f:
        text = f.read()
    body = re.search(r"struct %s \{.*?constexpr float c\[n\] = \{(.*?)\};" % name, text, re.S).group(1)
    c = [np.float64(np.float32(v.strip().rstrip("f"))) for v in body.split(",")]
    assert len(c) == int(re.search(r"struct %s \{\s*static constexpr int n = (\d+)" % name, text).group(1))
    return c, float(re.search(r"kSmallStrain = ([0-9.]+)f", text).group(1))


@pytest.mark.parametrize("name,exact", [
    ("PolyY", lambda m: -np.expm1(-0.5 * np.log1p(m))),
    ("PolyQ", lambda m: np.log1p(m) / (2.0 * (1.0 + m))),
])
def test_polynomial_is_as_close_as_stated(name, exact):
    c, bound = coefficients(name)
    t = np.linspace(-1.0, 1.0, 200_001)
    m = np.concatenate([bound * t, bound * np.sign(t) * 10.0 ** (-9.0 * np.abs(t))])
    m = m[m != 0.0]
    p = np.zeros_like(m)
    for k in reversed(c):
        p = p * m + k
    err = np.abs(m * p / exact(m) - 1.0)
    assert err.max() < 1.5e-8, "%s: %.2e at m = %.4f" % (name, err.max(), m[np.argmax(err)])
