"""Graphs with many edges a vertex, whose light edges are picked by a low rank in a
small sample: bit-exact at several seeds, and a batch of them well below the
round loop's time whatever the sample drew."""
from __future__ import annotations

import time

import numpy as np
import pytest

import oracle
from gpu_util import assert_parity, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_04865_gb300 import build_lib
    build_lib.build()


def make(n, m, seed):
    rng = np.random.default_rng(seed)
    return (rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32),
            rng.standard_normal(m).astype(np.float32))


@pytest.mark.parametrize("n,m", [(2, 8193), (60, 9000), (100, 400000), (1000, 60000), (2000, 524288), (4000, 400000),
                                 (3000, 1 << 20), (10000, 2000000), (400, 3000000)])
def test_one_graph(n, m):
    for seed in range(3):
        assert_parity(n, *make(n, m, seed), 0)


def batch(n, m, G, seed):
    s, d, w = make(n, m * G, seed)
    off = np.arange(G + 1, dtype=np.int64)
    return off * n, off * m, s, d, w


@pytest.mark.parametrize("n,m,G", [(2000, 524288, 3), (1000, 60000, 20), (300, 9000, 200)])
def test_batches(n, m, G):
    from paper_2110_04865_gb300 import api
    voff, eoff, s, d, w = batch(n, m, G, G)
    got = api.compute_batched(voff, eoff, to_dev(s), to_dev(d), to_dev(w))
    for a, b in zip(got, oracle.kruskal_batched(voff, eoff, s, d, w, 0)):
        assert np.array_equal(a.cpu().numpy(), b)


@pytest.mark.parametrize("seed", range(3))
def test_time_of_a_batch(seed):
    import torch
    from paper_2110_04865_gb300 import _abi, api
    voff, eoff, s, d, w = batch(2000, 524288, 40, seed)
    arrays = [to_dev(a) for a in (s, d, w)]

    def best():
        ts = []
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            api.compute_batched(voff, eoff, *arrays)
            ts.append(time.perf_counter() - t0)
        return min(ts[1:])

    now = best()
    old = _abi.msf_get_option(_abi.OPT_BUILD)
    try:
        _abi.msf_set_option(_abi.OPT_BUILD, 1)  # the round loop over the union's CSR
        loop = best()
    finally:
        _abi.msf_set_option(_abi.OPT_BUILD, old)
    assert now < 0.4 * loop  # (with one of 256 samples as the threshold 0.6 to 0.8)
