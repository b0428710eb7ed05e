"""Trees and graphs with few more edges than vertices, kept on the device: the
forest is the oracle's, the rounds are the loop's, and the call is no slower."""
from __future__ import annotations

import time

import numpy as np
import pytest

import oracle
from gpu_util import to_dev

pytestmark = pytest.mark.gpu

N = 3200000  # of edges, beyond those that are always counted in one class


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_04865_gb300 import build_lib
    build_lib.build()


def edges(kind):
    rng = np.random.default_rng(2)
    v = np.arange(N - 1, dtype=np.int32)
    if kind == "path":
        p = rng.permutation(N).astype(np.int32)
        return p[v], p[v + 1], v.astype(np.float32)
    if kind == "tree":
        return (rng.random(N - 1) * (v + 1)).astype(np.int32), v + 1, rng.random(N - 1).astype(np.float32)
    m = int(N * {"1.59": 1.59, "1.61": 1.61}[kind])
    return (rng.integers(0, N, m).astype(np.int32), rng.integers(0, N, m).astype(np.int32),
            rng.random(m).astype(np.float32))


@pytest.mark.parametrize("kind", ["path", "tree", "1.59", "1.61"])
def test_forest_rounds_and_time(kind):
    import torch
    from paper_2110_04865_gb300 import _abi, api
    s, d, w = edges(kind)
    g = api.Graph(N, *(to_dev(a) for a in (s, d, w)))

    def run():
        out = g.compute()
        ts = []
        for _ in range(5):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            g.compute()
            ts.append(time.perf_counter() - t0)
        return out, g.stats().rounds, g.stats().forest_edges, sorted(ts)[2]

    got, rounds, count, t = run()
    for a, b in zip(got, oracle.kruskal(N, s, d, w, 0)):
        assert np.array_equal(a.cpu().numpy(), np.atleast_1d(b))
    old = _abi.msf_get_option(_abi.OPT_COMPACT_TAU)
    try:
        _abi.msf_set_option(_abi.OPT_COMPACT_TAU, 0.25)  # the loop over the CSR
        _, loop_rounds, loop_count, loop_t = run()
    finally:
        _abi.msf_set_option(_abi.OPT_COMPACT_TAU, old)
    g.free()
    assert (rounds, count) == (loop_rounds, loop_count)
    assert t < 1.15 * loop_t
