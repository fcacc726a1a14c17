"""The bound behind the binary64 form's update terms in binary32, emulated on the
CPU: the coefficients at the largest magnitude that the kernels' rule admits,
every one of 62 columns, elements and coefficients cut to 24 bits as low_word
does, four chains of binary32 multiply-adds.  What is off stays within 2^-56 of
the update's scale, an eighth of the binary64 rounding (2^-53) of the exact
terms beside them.
"""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _constant(name):
    src = open(os.path.join(ROOT, "paper_2201_07498_gb300", "csrc", "te_reorth.cu")).read()
    return int(re.search(r"constexpr int %s = (-?\d+)" % name, src).group(1))


def _cut(x):  # to 24 significant bits, towards zero
    f, e = np.frexp(x)
    return np.ldexp(np.trunc(np.ldexp(f, 24)), e - 24)


def _terms(V, c):
    f = np.zeros((V.shape[0], 4), dtype=np.float32)
    Vl, cl = _cut(V), _cut(c)
    for j in range(V.shape[1]):  # (a product of 24-bit numbers is exact in binary64)
        u = j % 4
        f[:, u] = (f[:, u].astype(np.float64) + Vl[:, j] * cl[j]).astype(np.float32)
    s = (f[:, 0] + f[:, 1]) + (f[:, 2] + f[:, 3])
    return s.astype(np.float64)


@pytest.mark.parametrize("kind", ["spread", "dense row"])
def test_error_at_the_threshold(kind):
    cols = 62
    rng = np.random.default_rng(1)
    n = 4 * cols if kind == "spread" else cols
    V = np.linalg.qr(rng.standard_normal((n, cols)))[0]
    if kind == "dense row":  # every column has its element of the row, of one sign
        V = np.abs(V) / np.linalg.norm(V, axis=1, keepdims=True)
    # an exponent below the threshold is taken: the coefficient's significand is
    # below 2, the scale's at least 1 and a column's bound up to twice its norm
    c = np.full(cols, np.nextafter(2.0 ** (_constant("LOW_BITS") + 2), 0.0))
    off = np.linalg.norm(_terms(V, c) - (V.astype(np.longdouble) @ c).astype(np.float64))
    if kind == "dense row":
        off /= np.sqrt(n)
    assert off <= 2.0 ** -56
