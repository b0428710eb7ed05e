"""Kept graphs whose edges are all self-loops (or, as a CSR, all on the diagonal):
an empty forest, every vertex its own component, and no slower than the loop."""
from __future__ import annotations

import time

import numpy as np
import pytest

from gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_04865_gb300 import build_lib
    build_lib.build()


def empty_forest(g, n, m):
    mk, lb, tt = (x.cpu().numpy() for x in g.compute())
    assert mk.shape == (m,) and not mk.any()
    assert np.array_equal(lb, np.arange(n)) and tt[0] == 0.0
    assert np.array_equal(g.components().cpu().numpy(), np.arange(n))
    return g.stats().rounds, g.stats().forest_edges


@pytest.mark.parametrize("csr", [False, True])
@pytest.mark.parametrize("n,m", [(1, 5), (100, 300), (5000, 70001), (1 << 20, 1 << 23)])
def test_self_loops(n, m, csr):
    import torch
    from paper_2110_04865_gb300 import _abi, api
    rng = np.random.default_rng(m)
    s = np.sort(rng.integers(0, n, m).astype(np.int32))
    w = rng.standard_normal(m).astype(np.float32)
    rp = to_dev(np.searchsorted(s, np.arange(n + 1)).astype(np.int64)) if csr else None
    g = api.Graph(n, None if csr else to_dev(s), to_dev(s), to_dev(w), rp)

    def median():
        ts = []
        for _ in range(7):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            g.compute()
            ts.append(time.perf_counter() - t0)
        return sorted(ts)[3]

    counts, t = empty_forest(g, n, m), median()
    old = _abi.msf_get_option(_abi.OPT_COMPACT_TAU)
    try:
        _abi.msf_set_option(_abi.OPT_COMPACT_TAU, 0.25)  # the loop over the CSR
        assert counts == empty_forest(g, n, m)
        assert t < median()
    finally:
        _abi.msf_set_option(_abi.OPT_COMPACT_TAU, old)
    g.free()
