"""The Jacobi phase on a T whose elements differ by more than binary64's normal
range: diagonal elements that no rotation touches come back as they are, in
their order by magnitude, however small they are beside the largest one (T is
held divided by its largest element's power of two, where they would be
subnormal or zero)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def te():
    import paper_2201_07498_gb300 as te
    te.load_library(build_if_missing=True)
    return te


@pytest.mark.parametrize("which", ["LM", "LA"])
@pytest.mark.parametrize("m", [2, 5, 22, 30, 48, 64])
def test_untouched_diagonal_is_exact(te, m, which):
    # powers from 2^500 down past 2^500 2^-1074, odd significands, either sign
    e = np.round(np.linspace(500.0, -600.0, m)).astype(int)
    alpha = np.ldexp(1.0 + np.arange(m) / 97.0, e) * np.where(np.arange(m) % 3 == 1, -1.0, 1.0)
    perm = np.random.default_rng(m).permutation(m)
    alpha = alpha[perm]
    theta, Y, _ = te.tridiag_eigs(torch.from_numpy(alpha).cuda(),
                                  torch.zeros(m + 1, dtype=torch.float64, device="cuda"), which)
    order = np.argsort(-np.abs(alpha) if which == "LM" else -alpha, kind="stable")
    assert np.array_equal(theta.cpu().numpy(), alpha[order])
    assert np.array_equal(Y.cpu().numpy(), np.eye(m)[:, order])


@pytest.mark.parametrize("m", [7, 31, 47])
def test_rotated_pair_beside_tiny_elements(te, m):
    # one coupled pair at 2^500; the others down to 2^-580, uncoupled
    alpha = np.ldexp(1.0 + np.arange(m) / 97.0, -530 - np.arange(m))
    alpha[0], alpha[1] = 2.0 ** 500, -(2.0 ** 500)
    beta = np.zeros(m + 1)
    beta[1] = 0.75 * 2.0 ** 500  # eigenvalues +-1.25 2^500
    theta, Y, _ = te.tridiag_eigs(torch.from_numpy(alpha).cuda(), torch.from_numpy(beta).cuda())
    theta = theta.cpu().numpy()
    assert np.all(np.abs(np.abs(theta[:2]) - 1.25 * 2.0 ** 500) <= 1e-15 * 2.0 ** 501)
    assert np.array_equal(theta[2:], alpha[2:])
