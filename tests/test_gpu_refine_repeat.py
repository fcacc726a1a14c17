"""A refined plan solves again to the same bits: the refinement's scratch lies over
the basis and the newest column and, for an odd number of vectors, the vectors
over the pass vector, all of which the next solve writes before it reads them.
Another start vector in between, so that nothing is right by being left over."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def te():
    import paper_2201_07498_gb300 as te
    te.load_library(build_if_missing=True)
    return te


@pytest.mark.parametrize("prec", ["fdf", "bdf", "8df"])
@pytest.mark.parametrize("reorth", ["full", "delayed"])
@pytest.mark.parametrize("order", ["keep", "degree"])
@pytest.mark.parametrize("n,K", [(255, 1), (257, 3), (3001, 7), (3001, 8), (70001, 5)])
def test_second_solve_equals_the_first(te, n, K, order, reorth, prec):
    A = synth.uniform_sym(n, 5, n + K)
    plan = te.Plan(te.CSR.from_host(A, prec), K, 2 * K + 1, prec, refine=True, order=order,
                   reorth=reorth)
    g = torch.Generator(device="cuda").manual_seed(n)
    v = [torch.rand(n, device="cuda", dtype=torch.float64, generator=g) for _ in range(2)]
    first = [t.clone() for t in plan.solve(v1=v[0], residuals=True)]
    plan.solve(v1=v[1], residuals=True)
    again = plan.solve(v1=v[0], residuals=True)
    for a, b in zip(first, again):
        assert torch.equal(a, b)
