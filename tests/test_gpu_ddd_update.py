"""The binary64 updates whose small coefficients are taken in binary32.

* The basis and T of the Lanczos phase satisfy their relations at the binary64
  level, at row counts around a tile and a few tiles per CTA, for both sweeps'
  forms: V^T V - I within m 2^-50 (a second-sweep dot and its correction
  per column, with a margin of 8 over 2^-53 each) and M V - V T - beta v_{m+1}
  e_m^T within (m + longest row) 2^-50 ||T|| per column.
* The elements are scaled by their columns' bounds, so a matrix times 2^k gives
  the same basis and T times 2^k, bit for bit, far from 1 as well.
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def te():
    import paper_2201_07498_gb300 as te
    te.load_library(build_if_missing=True)
    return te


def _lanczos(te, A, m, reorth, k=0):
    B = synth.CSR(A.n, A.row_ptr, A.col, np.ldexp(A.val, k))
    a, b, V, _ = te.lanczos(te.CSR.from_host(B, "ddd"), m, "ddd", seed=3, reorth=reorth)
    return a.numpy(), b.numpy(), V.cpu().numpy()


@pytest.mark.parametrize("reorth", ["full", "delayed"])
@pytest.mark.parametrize("n,m", [(255, 40), (257, 41), (5000, 64), (300001, 24)])
def test_lanczos_relations_hold(te, n, m, reorth):
    A = synth.uniform_sym(n, 6, n)
    a, b, V = _lanczos(te, A, m, reorth)
    T = np.diag(a) + np.diag(b[1:m], 1) + np.diag(b[1:m], -1)
    tn = np.linalg.norm(T, 2)
    u = 2.0 ** -50
    assert np.max(np.abs(V.T @ V - np.eye(m))) <= m * u
    rows = np.repeat(np.arange(n), np.diff(A.row_ptr))
    MV = np.zeros_like(V)
    np.add.at(MV, rows, A.val[:, None] * V[A.col])
    R = (MV - V @ T)[:, :m - 1]
    longest = int(np.max(np.diff(A.row_ptr)))
    assert np.max(np.linalg.norm(R, axis=0)) <= (m + longest) * u * tn


@pytest.mark.parametrize("reorth", ["full", "delayed"])
@pytest.mark.parametrize("k", [-300, -31, 31, 300])
def test_lanczos_scales_exactly(te, k, reorth):
    A = synth.rmat_sym(12, 8, 5)
    a0, b0, V0 = _lanczos(te, A, 30, reorth)
    a, b, V = _lanczos(te, A, 30, reorth, k)
    assert np.array_equal(V, V0)
    assert np.array_equal(a, np.ldexp(a0, k)) and np.array_equal(b, np.ldexp(b0, k))
