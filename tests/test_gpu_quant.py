"""The quantisers where the integer and binary32 forms hand over to the exact
ones: values within a few binary64 units and within binary32's error of every
tie of a code, in rows of arbitrary scale, and scales whose binary32 rounding is
a near tie; both ends of the ranges, zeros, subnormals.  Bit for bit against the
oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def te():
    import paper_2201_07498_gb300 as te
    te.load_library(build_if_missing=True)
    return te


def _near(x):
    """x and its neighbours at binary64's and binary32's resolutions."""
    out = [x]
    for k in (-52, -51, -44, -30, -24, -22, -21, -20, -19, -18):
        out += [x * (1 + 2.0 ** k), x * (1 - 2.0 ** k)]
    return np.concatenate(out)


def _csr(rows):
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    val = np.concatenate(rows)
    n = max(len(rows), max(len(r) for r in rows))
    rp = np.concatenate([rp, np.full(n - len(rows), rp[-1])])
    col = np.concatenate([np.arange(len(r)) for r in rows]).astype(np.int32)
    return synth.CSR(n, rp, col, val)


def _check(te, A):
    csr = te.CSR.from_host(A, "ddd")
    codes, _ = te.quantize(csr, "bf16")
    assert np.array_equal(codes.cpu().numpy().view(np.uint16), oracle.round_bf16(A.val)[0])
    with np.errstate(over="ignore"):
        f32 = A.val.astype(np.float32)
    assert np.array_equal(te.quantize(csr, "f32")[0].cpu().numpy(), f32)
    c8, sc = te.quantize(csr, "e4m3")
    w8, wsc, _ = oracle.quantize_e4m3_rows(A)
    assert np.array_equal(sc.cpu().numpy(), wsc)
    # (a row below 2^-149 * 448 has scale 0: its codes are undefined)
    live = np.repeat(wsc, np.diff(A.row_ptr)) > 0
    assert np.array_equal(c8.cpu().numpy()[live], w8[live])


def test_ties_of_e4m3_codes(te):
    rng = np.random.default_rng(2)
    grid = np.array([m * 2.0 ** -9 for m in range(8)] +
                    [(1 + m / 8) * 2.0 ** (e - 7) for e in range(1, 16) for m in range(8)][:-1])
    mids = _near((grid[:-1] + grid[1:]) / 2)
    rows = []
    for _ in range(60):
        top = np.exp2(rng.uniform(-60, 60)) * 448.0
        s = float(np.float32(top / 448.0))
        rows.append(np.concatenate([[top, -top, 0.0], s * mids, -s * mids]))
        rows[-1] = rows[-1][np.abs(rows[-1]) <= top]
    _check(te, _csr(rows))


def test_ties_of_scales(te):
    """The largest magnitude of a row at and around 448 (s + ulp / 2)."""
    rng = np.random.default_rng(3)
    s = np.exp2(rng.uniform(-40, 40, 200)).astype(np.float32)
    mid = (s.astype(np.float64) + np.nextafter(s, np.float32(np.inf)).astype(np.float64)) / 2
    tops = np.concatenate([_near(448.0 * mid), 448.0 * np.exp2(np.arange(-50.0, 50.0))])
    _check(te, _csr([np.array([t, t * 0.3, -t * 0.01]) for t in tops]))


def test_ends_of_the_ranges(te):
    f32 = np.array([1.5, 1.0 + 2.0 ** -24, 1.0 + 3 * 2.0 ** -24, 2.0 ** -126, 2.0 ** -126 - 2.0 ** -160,
                    2.0 ** -149, 2.0 ** -150, 2.0 ** -133, 2.0 ** -134, 3e38,
                    2.0 ** 128 - 2.0 ** 103, 2.0 ** 127 * 1.998, 0.0, -0.0, 5e-324, 1e-310])
    rows = [np.array([x, -x]) for x in f32] + [f32, -f32, np.zeros(3)]
    bf = (np.arange(0x0001, 0x0400, dtype=np.uint32) << 16).view(np.float32).astype(np.float64)
    rows.append(_near((bf[:-1] + bf[1:]) / 2))
    _check(te, _csr(rows))
