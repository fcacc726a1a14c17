"""The SpMV's two forms (eight entries per lane in flight, or four and more
CTAs): rows by degree take the second from 72 (binary64) or 128 (binary32)
slices of 32 rows per SM on, the caller's order from 256 or 512.  Row counts on
either side of each, rows of 0 ... 20 entries: two steps of the Lanczos phase agree
between the orders within the summation bound of a row (20 products) and of the
dots' own rounding."""
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


@pytest.mark.parametrize("prec,per_sm,u", [("ddd", 72, 2.0 ** -53), ("fdf", 128, 2.0 ** -24),
                                           ("ddd", 256, 2.0 ** -53), ("fdf", 512, 2.0 ** -24)])
@pytest.mark.parametrize("side", [-3, 3])
def test_forms_agree(te, prec, per_sm, u, side):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = (per_sm + side) * sms * 32 + 7
    A = synth.uniform_sym(n, 2, 9)
    A = A if prec == "ddd" else A.with_f32_values()
    csr = te.CSR.from_host(A, prec)
    a, b, V, _ = te.lanczos(csr, 3, prec, seed=2, order="keep")
    a2, b2, V2, _ = te.lanczos(csr, 3, prec, seed=2, order="degree")
    tn = float(torch.max(a.abs()) + 2 * torch.max(b.abs()))
    # per step: 20 products of a row, the stored vector's rounding, two sweeps
    tol = 3 * 64 * u
    assert float((a - a2).abs().max()) <= tol * tn
    assert float((b - b2).abs().max()) <= tol * tn
    assert float((V - V2).norm(dim=0).max()) <= tol * tn / float(b[1:3].min())
