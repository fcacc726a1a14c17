"""The binary64 Ritz vectors taken in digits on the tensor pipe.

U = V Y from the Lanczos phase's own V and Y, in extended precision on the CPU,
at the edges of the kernel's steps of 16 columns and tiles of 16 outputs and of
the rule that takes it (m times K, rounded up to 8, from 80 on), for both storage
forms (by columns, and by rows under a relabelled order).  Per
element: m + 4 roundings of the products' magnitudes (V's own scaling, a binary64
sum; the digits make one), and 2^-57 of the two bounds' product (61-bit digits
of both factors, 2^-59 left out, m <= 64 terms each with its own cut).
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


def _check(te, A, K, m, order):
    csr = te.CSR.from_host(A, "ddd")
    a, b, V, _ = te.lanczos(csr, m, "ddd", seed=3, order=order)
    theta, Y, _ = te.tridiag_eigs(a.cuda(), b.cuda())
    ev, U, _ = te.topk_eigs(csr, K, m, "ddd", seed=3, order=order)
    assert np.array_equal(np.asarray(ev), theta.cpu().numpy()[:K])
    V = V.cpu().numpy().astype(np.longdouble)
    Y = Y.cpu().numpy()[:, :K].astype(np.longdouble)
    U = U.cpu().numpy()
    ref = V @ Y
    tol = (m + 4) * 2.0 ** -53 * (np.abs(V) @ np.abs(Y))
    tol += 2.0 ** -57 * np.abs(V).max(1, keepdims=True) * np.abs(Y).max(0, keepdims=True)
    assert np.all(np.abs(U - ref) <= tol)


@pytest.mark.parametrize("order", ["keep", "degree"])
@pytest.mark.parametrize("n,K,m", [(999, 8, 9), (1000, 8, 10), (255, 1, 16), (257, 7, 17), (1000, 16, 32), (1001, 17, 33),
                                   (4097, 33, 48), (2503, 64, 64), (70001, 15, 31)])
def test_ritz_vectors(te, n, K, m, order):
    _check(te, synth.uniform_sym(n, 6, n), K, m, order)


def test_wide_rows_and_scales(te):
    A = synth.rmat_sym(12, 8, 5)
    for k in (-300, 0, 300):  # the basis' columns carry the matrix' scale
        B = synth.CSR(A.n, A.row_ptr, A.col, np.ldexp(A.val, k))
        _check(te, B, 9, 24, "degree")
