"""Gram-Schmidt's second sweep where beta is far below |alpha|: M = I + 2^-k B.

What the first sweep leaves along the basis grows against the vector as beta
shrinks (about 2^(k - 53) of it), so that the second sweep's coefficients go from
the rounding level, where their terms are taken in binary32, through the
threshold to where they have to be binary64.  V^T V - I stays within m 2^-50 (a
second-sweep dot and its correction per column, with a margin of 8 over 2^-53
each) and M V - V T - beta v_{m+1} e_m^T within (m + longest row) 2^-50 ||T|| per
column, in both forms and whatever k.  The entries are exact: B has no diagonal.
More tiles of 256 rows than the GPU has SMs: with fewer every term is binary64.
A matrix times a power of two gives the same basis there too, bit for bit.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

N = 80_003  # 313 tiles


@pytest.fixture(scope="module")
def te():
    import paper_2201_07498_gb300 as te
    te.load_library(build_if_missing=True)
    return te


def _near_identity(n, k, seed):
    B = synth.uniform_sym(n, 6, seed)
    rows = np.repeat(np.arange(n), np.diff(B.row_ptr))
    off = rows != B.col
    scale = 2.0 ** -(k + 3)  # ||B|| is about 7
    r = np.concatenate([rows[off], np.arange(n)])
    c = np.concatenate([B.col[off], np.arange(n)])
    v = np.concatenate([B.val[off] * scale, np.ones(n)])
    return synth.from_triplets(n, r, c, v)


@pytest.mark.parametrize("reorth", ["full", "delayed"])
@pytest.mark.parametrize("k", [0, 2, 4, 6, 7, 8, 9, 10, 11, 12, 14, 17, 20, 22, 24, 26, 28, 30, 32,
                               34, 36])
def test_basis_stays_orthonormal(te, k, reorth):
    n, m = N, 30
    A = _near_identity(n, k, 5)
    a, b, V, restarts = te.lanczos(te.CSR.from_host(A, "ddd"), m, "ddd", seed=3, reorth=reorth)
    a, b, V = a.numpy(), b.numpy(), V.cpu().numpy()
    assert restarts == 0
    u = 2.0 ** -50
    assert np.max(np.abs(V.T @ V - np.eye(m))) <= m * u
    T = np.diag(a) + np.diag(b[1:m], 1) + np.diag(b[1:m], -1)
    rows = np.repeat(np.arange(n), np.diff(A.row_ptr))
    MV = np.zeros_like(V)
    np.add.at(MV, rows, A.val[:, None] * V[A.col])
    R = (MV - V @ T)[:, :m - 1]
    longest = int(np.max(np.diff(A.row_ptr)))
    assert np.max(np.linalg.norm(R, axis=0)) <= (m + longest) * u * np.linalg.norm(T, 2)


@pytest.mark.parametrize("reorth", ["full", "delayed"])
@pytest.mark.parametrize("k", [-300, 31, 300])
def test_scales_exactly(te, k, reorth):
    A = synth.uniform_sym(N, 6, 5)
    B = synth.CSR(N, A.row_ptr, A.col, np.ldexp(A.val, k))
    a0, b0, V0, _ = te.lanczos(te.CSR.from_host(A, "ddd"), 30, "ddd", seed=3, reorth=reorth)
    a, b, V, _ = te.lanczos(te.CSR.from_host(B, "ddd"), 30, "ddd", seed=3, reorth=reorth)
    assert np.array_equal(V.cpu().numpy(), V0.cpu().numpy())
    assert np.array_equal(a.numpy(), np.ldexp(a0.numpy(), k))
    assert np.array_equal(b.numpy(), np.ldexp(b0.numpy(), k))
