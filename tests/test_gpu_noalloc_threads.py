"""te_spmv_noalloc from more host threads than it has status slots (64), all on one
stream: every call returns its own status, errors of one never reach another,
and what it wrote is its own matrix's product."""
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def te():
    import paper_2201_07498_gb300 as te
    te.load_library(build_if_missing=True)
    return te


def test_each_thread_gets_its_own_status(te):
    threads, calls, n = 80, 5, 3000
    rng = np.random.default_rng(4)
    rp = torch.arange(0, 4 * n + 1, 4, dtype=torch.int64, device="cuda")
    val = torch.from_numpy(rng.integers(1, 9, 4 * n).astype(np.float64)).cuda()
    x = torch.from_numpy(rng.integers(-9, 9, n).astype(np.float64)).cuda()
    cases = []
    for t in range(threads):
        col = rng.integers(0, n, 4 * n)
        want = (val.cpu().numpy() * x.cpu().numpy()[col]).reshape(n, 4).sum(1)
        if t % 3 == 0:
            col[rng.integers(4 * n)] = n  # outside [0, n): the kernel reports it
        col = torch.from_numpy(col.astype(np.int32)).cuda()
        cases.append((te.CSR(n, rp, col, val), want,
                      torch.empty(n, dtype=torch.float64, device="cuda")))
    torch.cuda.synchronize()
    bad = []

    def work(t):
        csr, want, y = cases[t]
        for _ in range(calls):
            try:
                te.spmv_noalloc(csr, x, y)
                if t % 3 == 0:
                    bad.append((t, "no error"))
            except Exception as e:
                if t % 3 != 0 or "column index" not in str(e):
                    bad.append((t, repr(e)))

    pool = [threading.Thread(target=work, args=(t,)) for t in range(threads)]
    for p in pool:
        p.start()
    for p in pool:
        p.join()
    assert not bad
    for t, (_, want, y) in enumerate(cases):
        if t % 3 != 0:  # (whole numbers: exact)
            assert np.array_equal(y.cpu().numpy(), want)
