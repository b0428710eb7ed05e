"""CSR input with long runs of empty rows (a few vertices of a large id range
have edges): the rows of the slots are found without walking the gaps, and the
edges are those of the oracle."""
from __future__ import annotations

import time

import numpy as np
import pytest

import oracle
from gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_04865_gb300 import build_lib
    build_lib.build()


def csr(n, s, d, w):
    """Symmetric CSR with sorted rows; slot weights are the edges'."""
    rows, cols, ww = np.concatenate([s, d]), np.concatenate([d, s]), np.concatenate([w, w])
    o = np.lexsort((cols, rows))
    rp = np.zeros(n + 1, np.int64)
    np.add.at(rp, rows[o].astype(np.int64) + 1, 1)
    return np.cumsum(rp), rows[o].astype(np.int32), cols[o].astype(np.int32), ww[o]


def edges(kind, n, k, m):
    """m edges among k vertices, which are spread over 0 .. n - 1."""
    rng = np.random.default_rng(k)
    ids = {"ends": np.concatenate([np.arange(k // 2), np.arange(n - (k - k // 2), n)]),
           "spread": np.arange(k) * (n // k) + 3,
           "runs": np.arange(k) + (np.arange(k) // 5) * (n // k)}[kind].astype(np.int64)
    s, d = (ids[rng.integers(0, k, m)] for _ in range(2))
    keep = s != d
    return s[keep].astype(np.int32), d[keep].astype(np.int32), rng.standard_normal(int(keep.sum())).astype(np.float32)


@pytest.mark.parametrize("kind", ["ends", "spread", "runs"])
@pytest.mark.parametrize("n,k,m", [(9000, 7, 400), (1 << 20, 700, 30000), (1 << 25, 1000, 60000)])
def test_forest_and_build_time(kind, n, k, m):
    import torch
    from paper_2110_04865_gb300 import api
    rp, rows, cols, w = csr(n, *edges(kind, n, k, m))
    arrays = to_dev(cols), to_dev(w), to_dev(rp)
    g = api.Graph(n, None, arrays[0], arrays[1], arrays[2])
    mk, lb, tt = g.compute()
    # a slot below the diagonal is no edge: a self-loop for the oracle
    omk, olb, otot = oracle.kruskal(n, np.where(rows < cols, rows, cols).astype(np.int32), cols, w, 0)
    assert np.array_equal(mk.cpu().numpy(), omk) and np.array_equal(lb.cpu().numpy(), olb)
    assert float(tt.cpu()[0]) == otot
    assert np.array_equal(g.components().cpu().numpy(), olb)
    g.free()
    # a search is some 25 loads of about a microsecond each; the vertices' own
    # passes take under a millisecond: far below the bound, a walk over 2^25
    # rows far above it
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    api.Graph(n, None, arrays[0], arrays[1], arrays[2]).free()
    assert time.perf_counter() - t0 < 0.05
