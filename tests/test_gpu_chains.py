"""Graphs whose hooks form long chains (paths and combs with weights that rise
or fall along them, trees of deep chains): the forests are the oracle's, and a
chain costs no more than a few times what a random graph of its size does."""
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


def chain(kind, n):
    v = np.arange(n - 1, dtype=np.int32)
    if kind == "rising":
        return v, v + 1, v.astype(np.float32)
    if kind == "falling":
        return v, v + 1, -v.astype(np.float32)
    if kind == "permuted":
        p = np.random.default_rng(n).permutation(n).astype(np.int32)
        return p[v], p[v + 1], v.astype(np.float32)
    # a comb: a chain along the even vertices, a tooth at each
    k = n // 2
    s = np.concatenate([2 * np.arange(k - 1), 2 * np.arange(k)]).astype(np.int32)
    d = np.concatenate([2 * np.arange(1, k), 2 * np.arange(k) + 1]).astype(np.int32)
    return s, d, np.concatenate([np.arange(k - 1), np.arange(k) + 0.5]).astype(np.float32)


def median(f):
    import torch
    f()
    ts = []
    for _ in range(7):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        f()
        ts.append(time.perf_counter() - t0)
    return sorted(ts)[3]


@pytest.mark.parametrize("kind", ["rising", "falling", "permuted", "comb"])
@pytest.mark.parametrize("n", [17, 18, 290, 5000, 14000, 20400, 60000, 300000])
def test_chains(kind, n):
    from paper_2110_04865_gb300 import api
    s, d, w = chain(kind, n)
    ref = oracle.kruskal(n, s, d, w, 0)
    arrays = [to_dev(a) for a in (s, d, w)]
    g = api.Graph(n, *arrays)
    copies = 3
    off = np.arange(copies + 1, dtype=np.int64)
    batch = api.compute_batched(off * n, off * len(s), *(a.repeat(copies) for a in arrays))
    for got in (api.compute(n, *arrays), g.compute()):
        for a, b in zip(got, ref):
            assert np.array_equal(a.cpu().numpy(), np.atleast_1d(b))
    assert np.array_equal(g.components().cpu().numpy(), ref[1])
    for a, b in zip(batch, ref):
        assert np.array_equal(a.cpu().numpy(), np.tile(np.atleast_1d(b), copies))
    g.free()


@pytest.mark.parametrize("kind", ["rising", "falling", "permuted"])
def test_chains_take_no_longer_than_random_graphs(kind):
    """A chain hooks in one round; a random tree takes several.  (Followed hop
    by hop the chain of 20 000 vertices took thirty times as long.)"""
    from paper_2110_04865_gb300 import api
    n = 20000
    rng = np.random.default_rng(1)
    tree = api.Graph(n, to_dev((rng.random(n - 1) * np.arange(1, n)).astype(np.int32)),
                     to_dev(np.arange(1, n, dtype=np.int32)), to_dev(rng.random(n - 1).astype(np.float32)))
    g = api.Graph(n, *(to_dev(a) for a in chain(kind, n)))
    assert median(g.compute) < 2 * median(tree.compute)
    g.free()
    tree.free()


@pytest.mark.parametrize("kind", ["rising", "falling", "permuted"])
@pytest.mark.parametrize("n", [40000, 100000])
def test_chains_take_no_longer_than_the_round_loop(kind, n):
    """(A threshold of its own selects the loop over the CSR.)"""
    from paper_2110_04865_gb300 import _abi, api
    g = api.Graph(n, *(to_dev(a) for a in chain(kind, n)))
    edges = median(g.compute)
    old = _abi.msf_get_option(_abi.OPT_COMPACT_TAU)
    try:
        _abi.msf_set_option(_abi.OPT_COMPACT_TAU, 0.25)
        loop = median(g.compute)
    finally:
        _abi.msf_set_option(_abi.OPT_COMPACT_TAU, old)
    g.free()
    assert edges < 1.15 * loop
