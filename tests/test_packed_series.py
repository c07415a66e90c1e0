"""The sine and cosine series of the transfer kernels, as written in the CUDA source: the packed forms carry the Taylor
coefficients, the cosine's packed and scalar forms are the same polynomial, and the truncation errors that the comments
state hold: the first omitted term at |x| = pi/2, which bounds an alternating series with falling terms."""
import math
import os
import re

import numpy as np
import pytest

SRC = open(os.path.join(os.path.dirname(__file__), "..", "paper_2412_10399_gb300", "csrc", "transfer.cu")).read()


def _horner(signature):
    """The constants of a Horner evaluation in t^2, ascending: p = c_n, then p = fma(p, t2, c)."""
    body = SRC[SRC.index(signature):]
    body = body[:body.index("return")]
    c = re.findall(r"p = (?:v3\(|dup\()?(-?\d+\.\d+)f", body) + re.findall(r"p, t2, (?:v3\(|dup\()?(-?\d+\.\d+)f", body)
    return [float(x) for x in c][::-1]


@pytest.mark.parametrize("signature,odd,terms", [("V3 sin_2pi(const V3& f)", 1, 6), ("V3 cos_2pi(const V3& f)", 0, 7),
                                                 ("float cos_2pi(float f)", 0, 7)])
def test_series_carry_the_taylor_coefficients(signature, odd, terms):
    coef = _horner(signature)
    assert len(coef) == terms
    for k, c in enumerate(coef):
        e = 2 * k + odd
        want = (-1) ** k * (2 * math.pi) ** e / math.factorial(e)
        assert abs(c - want) <= 1e-15 * abs(want)


@pytest.mark.parametrize("signature,odd,f", [("V3 sin_2pi(const V3& f)", 1, math.sin),
                                             ("V3 cos_2pi(const V3& f)", 0, math.cos)])
def test_stated_truncation_errors(signature, odd, f):
    coef = _horner(signature)
    power = 2 * len(coef) + odd
    head = SRC[:SRC.index(signature)]
    text = re.sub(r"\s*//\s*", " ", head[head.rindex("Taylor series of " + ("sin" if odd else "cos")):])
    m = re.search(r"\(pi/2\)\^(\d+) / (\d+)! = ([0-9.e-]+)[,.]", text)
    assert int(m.group(1)) == int(m.group(2)) == power
    term = (math.pi / 2) ** power / math.factorial(power)
    assert term <= float(m.group(3)) <= 1.1 * term
    t = np.linspace(0.0, 0.25, 2001)
    s = sum(c * t ** (2 * k + odd) for k, c in enumerate(coef))
    assert np.abs(s - np.array([f(2 * math.pi * x) for x in t])).max() <= float(m.group(3))
