"""msf_connected_components over the edges: labels and rounds are those of the
loop over the CSR (which a round limit below the default selects) and of the
oracle, at the sizes where pages, blocks and the bitmap's place change."""
from __future__ import annotations

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


def check(n, s, d):
    from paper_2110_04865_gb300 import _abi, api
    w = np.ones(len(s), np.float32)
    g = api.Graph(n, to_dev(s), to_dev(d), to_dev(w))
    old = _abi.msf_get_option(_abi.OPT_ROUND_LIMIT)
    try:
        lb = [g.components().cpu().numpy() for _ in range(2)]
        rounds = g.stats().cc_rounds
        _abi.msf_set_option(_abi.OPT_ROUND_LIMIT, 63)
        ref = g.components().cpu().numpy()
        assert rounds == g.stats().cc_rounds
    finally:
        _abi.msf_set_option(_abi.OPT_ROUND_LIMIT, old)
        g.free()
    assert np.array_equal(lb[0], ref) and np.array_equal(lb[1], ref)
    assert np.array_equal(ref, oracle.kruskal(n, s, d, w, 0)[1])


@pytest.mark.parametrize("n,m", [(1, 0), (1, 3), (2, 1), (129, 127), (1000, 1023), (1024, 1025), (5000, 3000),
                                 (155648, 155649), (300000, 150001), (1835008, 3000000), (1835009, 900001),
                                 (2500000, 4000003), (40000, 2600001)])
def test_random(n, m):
    rng = np.random.default_rng(n + m)
    check(n, rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32))


@pytest.mark.parametrize("shape", ["path", "path back", "path shuffled", "hub high", "blocks", "lattice"])
def test_shapes(shape):
    rng = np.random.default_rng(5)
    n = 120001
    a = np.arange(n - 1, dtype=np.int32)
    s, d = a, a + 1
    if shape == "path back":
        s, d = d[::-1].copy(), s[::-1].copy()
    elif shape == "path shuffled":
        ids = rng.permutation(n).astype(np.int32)
        s, d = ids[:-1].copy(), ids[1:].copy()
    elif shape == "hub high":  # every edge offers to one root
        m = 500000
        s, d = np.full(m, n - 1, np.int32), rng.integers(0, n, m).astype(np.int32)
    elif shape == "blocks":  # no giant tree
        m = 700000
        s = (rng.integers(0, n, m) // 16 * 16).astype(np.int32)
        d = np.minimum(s + rng.integers(0, 16, m), n - 1).astype(np.int32)
    elif shape == "lattice":
        k = 48
        v = np.arange(k ** 3).reshape(k, k, k)
        s = np.concatenate([v[1:].ravel(), v[:, 1:].ravel(), v[:, :, 1:].ravel()]).astype(np.int32)
        d = np.concatenate([v[:-1].ravel(), v[:, :-1].ravel(), v[:, :, :-1].ravel()]).astype(np.int32)
        n = k ** 3
    check(n, s, d)


def test_small_sparse_graphs():
    """Many trees and rounds, vertex 0 often no root, the last page of the
    vertices partly filled: labels and rounds of the step oracle."""
    from oracle import as_cc
    from paper_2110_04865_gb300 import api
    rng = np.random.default_rng(0)
    for _ in range(120):
        n = int(rng.integers(2, 3000))
        m = int(rng.integers(1, 3 * n))
        s, d = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
        g = api.Graph(n, to_dev(s), to_dev(d), to_dev(np.ones(m, np.float32)))
        lb = g.components().cpu().numpy()
        rounds = g.stats().cc_rounds
        g.free()
        ref = as_cc.as_cc(n, s, d)
        assert np.array_equal(lb, ref["labels"]) and rounds == ref["rounds"]
