"""The delayed form's binary64 dots taken in digits on the tensor pipe.

Digits start at 8 columns and 6 tiles of 256 rows per CTA (912 tiles on 152 SMs),
in groups of 8 columns:

* around these edges, and with a last tile of one row, V^T V - I stays within
  m 2^-50 and M V - V T within (m + longest row) 2^-50 ||T|| per column (a
  second-sweep dot and its correction per column, with a margin of 8 over 2^-53);
* rows that grow by 2^60 from the first tile to the last (the vectors' bound grows
  on the way) keep the same relations;
* a matrix times 2^k gives the same basis and T times 2^k, bit for bit;
* an infinity or NaN in the matrix reaches every alpha and leaves the basis (whose
  vectors are drawn again) orthonormal, as below 8 columns.
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

EDGE = 911 * 256  # 911 full tiles


@pytest.fixture(scope="module")
def te():
    import paper_2201_07498_gb300 as te
    te.load_library(build_if_missing=True)
    return te


def _lanczos(te, A, m, k=0):
    B = synth.CSR(A.n, A.row_ptr, A.col, np.ldexp(A.val, k))
    a, b, V, _ = te.lanczos(te.CSR.from_host(B, "ddd"), m, "ddd", seed=3, reorth="delayed")
    return a.numpy(), b.numpy(), V.cpu().numpy()


def _relations(A, m, a, b, V):
    T = np.diag(a) + np.diag(b[1:m], 1) + np.diag(b[1:m], -1)
    u = 2.0 ** -50
    assert np.max(np.abs(V.T @ V - np.eye(m))) <= m * u
    rows = np.repeat(np.arange(A.n), np.diff(A.row_ptr))
    R = np.empty((A.n, m))
    for j in range(m):
        R[:, j] = np.bincount(rows, A.val * V[A.col, j], A.n)
    R = (R - V @ T)[:, :m - 1]
    longest = int(np.max(np.diff(A.row_ptr)))
    assert np.max(np.linalg.norm(R, axis=0)) <= (m + longest) * u * np.linalg.norm(T, 2)


@pytest.mark.parametrize("n,m", [(EDGE, 20), (EDGE + 1, 9), (EDGE + 1, 18), (EDGE + 1, 27),
                                 (EDGE + 1, 64), (400_003, 34)])
def test_relations_hold(te, n, m):
    A = synth.uniform_sym(n, 4, n + m)
    _relations(A, m, *_lanczos(te, A, m))


def test_growing_rows(te):
    n, m = EDGE + 257, 20
    A = synth.uniform_sym(n, 4, 11)
    d = np.floor(60.0 * np.arange(n) / n).astype(int) // 2
    rows = np.repeat(np.arange(n), np.diff(A.row_ptr))
    A = synth.CSR(n, A.row_ptr, A.col, np.ldexp(A.val, d[rows] + d[A.col]))
    _relations(A, m, *_lanczos(te, A, m))


@pytest.mark.parametrize("k", [-300, 300])
def test_scales_exactly(te, k):
    A = synth.uniform_sym(EDGE + 1, 4, 5)
    a0, b0, V0 = _lanczos(te, A, 20)
    a, b, V = _lanczos(te, A, 20, k)
    assert np.array_equal(V, V0)
    assert np.array_equal(a, np.ldexp(a0, k)) and np.array_equal(b, np.ldexp(b0, k))


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_not_finite(te, bad):
    A = synth.uniform_sym(EDGE + 1, 4, 7)
    v = A.val.copy()
    v[12345] = bad
    m = 20
    a, b, V = _lanczos(te, synth.CSR(A.n, A.row_ptr, A.col, v), m)
    assert not np.isfinite(a).any() and np.isfinite(b).all()
    assert np.max(np.abs(V.T @ V - np.eye(m))) <= m * 2.0 ** -50
