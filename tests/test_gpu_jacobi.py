"""The Jacobi phase at the orders where its launch changes (one CTA, clusters of
four and of eight, the warp that takes the last elements of m > 60) against
the oracle, and its scaling: T times a power of two, up to the ends of
binary64's range, gives the same vectors and sweeps and the scaled values,
bit for bit."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def te():
    import paper_2201_07498_gb300 as te
    te.load_library(build_if_missing=True)
    return te


def _t(m):
    rng = np.random.default_rng(1000 + m)
    return rng.standard_normal(m), np.concatenate([[0.0], np.abs(rng.standard_normal(m))])


def _eigs(te, alpha, beta, which="LM"):
    theta, Y, sweeps = te.tridiag_eigs(torch.from_numpy(alpha).cuda(),
                                       torch.from_numpy(beta).cuda(), which)
    return theta.cpu().numpy(), Y.cpu().numpy(), sweeps


@pytest.mark.parametrize("m", [4, 5, 21, 22, 23, 24, 36, 37, 60, 61, 63])
def test_jacobi_at_launch_edges(te, m):
    alpha, beta = _t(m)
    T = np.diag(alpha) + np.diag(beta[1:m], 1) + np.diag(beta[1:m], -1)
    theta, Y, _ = _eigs(te, alpha, beta)
    th_ref, _, _, _ = oracle.jacobi(T)
    idx = oracle.select_topk(th_ref, m, oracle.LARGEST_MAGNITUDE)
    tn = np.linalg.norm(T)
    assert np.max(np.abs(theta - th_ref[idx])) <= 1e-13 * tn
    assert np.max(np.abs(T @ Y - Y * theta)) <= 1e-13 * tn
    assert np.max(np.abs(Y.T @ Y - np.eye(m))) <= 1e-13


@pytest.mark.parametrize("m", [12, 30, 48])
@pytest.mark.parametrize("k", [-960, -40, 40, 1000])
def test_jacobi_scales_exactly(te, m, k):
    alpha, beta = _t(m)
    th0, Y0, s0 = _eigs(te, alpha, beta)
    th, Y, s = _eigs(te, np.ldexp(alpha, k), np.ldexp(beta, k))
    assert s == s0
    assert np.array_equal(Y, Y0)
    assert np.array_equal(th, np.ldexp(th0, k))


def test_jacobi_of_zero_and_diagonal(te):
    m = 17
    th, Y, _ = _eigs(te, np.zeros(m), np.zeros(m + 1))
    assert np.array_equal(th, np.zeros(m)) and np.array_equal(Y, np.eye(m))
    d = np.arange(1.0, m + 1)
    th, Y, _ = _eigs(te, d, np.zeros(m + 1))
    assert np.array_equal(th, d[::-1]) and np.array_equal(Y, np.eye(m)[:, ::-1])
