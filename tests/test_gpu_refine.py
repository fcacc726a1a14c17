"""The refinement's products of several vectors at a time: K around the group
sizes (1, 2, 4, 8 vectors), cut rows of a few and of many pieces, rows without
entries, rows relabelled or not, a matrix so dense that the cut rows' sums of
several vectors do not fit the basis.  Against the Rayleigh quotients and the
residuals that numpy computes from the returned vectors in binary64: each a sum
over the rows of sums over a row, so within 4 (longest row + 64) 2^-53 ||M||_inf
(the blocks' partial sums are short chains)."""
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


def _matrix(kind):
    rng = np.random.default_rng(7)
    if kind == "dense":  # every row cut, many pieces
        n = 900
        d = rng.uniform(0, 1, (n, n))
        return synth.from_dense(d + d.T)
    n = 20000  # a hub row, rows of 65 ... 300 entries, every fourth row empty
    live = np.arange(n)[np.arange(n) % 4 != 0]
    r, c = [np.full(len(live) - 1, live[0])], [live[1:]]
    for i in live[1:60]:
        k = int(rng.integers(65, 300))
        r.append(np.full(k, i))
        c.append(rng.choice(live, k, replace=False))
    r.append(rng.choice(live, 60000))
    c.append(rng.choice(live, 60000))
    r, c = np.concatenate(r), np.concatenate(c)
    v = rng.uniform(0, 1, len(r))
    return synth.from_triplets(n, np.concatenate([r, c]), np.concatenate([c, r]),
                               np.concatenate([v, v]))


@pytest.mark.parametrize("order", ["keep", "degree"])
@pytest.mark.parametrize("K", [1, 2, 3, 5, 8, 9, 15])
@pytest.mark.parametrize("kind", ["hubs", "dense"])
def test_refined_values_are_the_quotients_of_the_vectors(te, kind, K, order):
    A = _matrix(kind)
    m = 2 * K + 2
    plan = te.Plan(te.CSR.from_host(A, "fdf"), K, m, "fdf", seed=1, refine=True, order=order)
    for _ in range(2):  # the second solve reuses the scratch
        ev, U, res = plan.solve(residuals=True)
    ev, U, res = ev.numpy(), U.cpu().numpy(), res.numpy()
    rows = np.repeat(np.arange(A.n), np.diff(A.row_ptr))
    Y = np.zeros_like(U)
    np.add.at(Y, rows, A.val[:, None] * U[A.col])
    uu = np.sum(U * U, axis=0)
    th = np.sum(U * Y, axis=0) / uu
    norm = np.max(np.bincount(rows, weights=np.abs(A.val), minlength=A.n))
    tol = 4 * (np.max(np.diff(A.row_ptr)) + 64) * 2.0 ** -53 * norm
    assert np.max(np.abs(ev - th)) <= tol
    true = np.linalg.norm(Y - U * ev, axis=0) / np.sqrt(uu)
    assert np.max(np.abs(res - true)) <= tol
