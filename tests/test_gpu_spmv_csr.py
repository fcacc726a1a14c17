"""te_spmv_noalloc at the edges of its chunks: entry counts around a chunk (and
around the 2048 chunks above which the rows are searched by a kernel of their
own), rows that end exactly at chunk boundaries, hub rows over more than a
warp of chunks, long runs of empty rows, and arrays that are not 16-byte
aligned; against the oracle within the summation bound of
test_zz_no_alloc.py."""
import numpy as np
import pytest
import torch

import oracle
import synth
from test_zz_no_alloc import _bound

pytestmark = pytest.mark.gpu

CH = {"ddd": 2048, "fdf": 4096}


@pytest.fixture(scope="module")
def te():
    import paper_2201_07498_gb300 as te
    te.load_library(build_if_missing=True)
    return te


def _lengths(kind, ch, rng):
    if kind == "one_short":
        return [3, ch - 4]  # nnz = chunk - 1
    if kind == "exact":
        return [0, 0, ch // 2, 0, ch // 2, 0]  # one full chunk, empty rows around
    if kind == "one_over":
        return [ch, 1]  # a row ends at the boundary, the next has one entry
    if kind == "aligned_rows":
        return [16, ch - 16, 0, ch, ch, 7]
    if kind == "hub":
        return list(rng.integers(0, 9, 500)) + [40 * ch + 5] + list(rng.integers(0, 9, 500))
    if kind == "empty_runs":
        return [5] + [0] * 70000 + [ch + 3] + [0] * 300 + [1] * 50 + [0] * 1000
    if kind == "searched":  # more than 2048 chunks
        return list(rng.integers(0, 40, 1000)) + [700 * ch] + list(rng.integers(0, 2 * ch, 1400))
    raise ValueError(kind)


@pytest.mark.parametrize("prec", ["ddd", "fdf"])
@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("kind", ["one_short", "exact", "one_over", "aligned_rows", "hub",
                                  "empty_runs", "searched"])
def test_noalloc_chunk_edges(te, kind, aligned, prec):
    rng = np.random.default_rng(len(kind))
    L = np.asarray(_lengths(kind, CH[prec], rng), dtype=np.int64)
    n, rp = len(L), np.concatenate([[0], np.cumsum(L)])
    nnz = int(rp[-1])
    dt = np.float64 if prec == "ddd" else np.float32
    col = rng.integers(0, n, nnz).astype(np.int32)
    val = rng.uniform(-1, 1, nnz).astype(dt)
    x = rng.uniform(-1, 1, n).astype(dt)

    def put(a):  # on the device, at an offset of one element unless aligned
        t = torch.zeros(len(a) + 4, dtype=torch.from_numpy(a).dtype, device="cuda")
        v = t[:len(a)] if aligned else t[1:1 + len(a)]
        v.copy_(torch.from_numpy(a))
        return v

    csr = te.CSR(n, torch.from_numpy(rp).cuda(), put(col), put(val))
    y = te.spmv_noalloc(csr, torch.from_numpy(x).cuda(), precision=prec).cpu().numpy()
    A = synth.CSR(n, rp, col, val.astype(np.float64))
    x64 = x.astype(np.float64)
    u = 2.0 ** -53 if prec == "ddd" else 2.0 ** -44
    assert np.all(np.abs(y - oracle.spmv(A, x64)) <= _bound(A, x64, u))
