"""Connected components of few vertices with very many edges: the labels of the
oracle and the loop's round count on both sides of the line up to which a
block collects the first offers, and no slower than the loop."""
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


def components(g, limit=None):
    """(labels, rounds, median seconds); a round limit of its own selects the loop."""
    import torch
    from paper_2110_04865_gb300 import _abi
    old = _abi.msf_get_option(_abi.OPT_ROUND_LIMIT)
    try:
        if limit:
            _abi.msf_set_option(_abi.OPT_ROUND_LIMIT, limit)
        labels = g.components().cpu().numpy()
        ts = []
        for _ in range(7):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            g.components()
            ts.append(time.perf_counter() - t0)
        return labels, g.stats().cc_rounds, sorted(ts)[3]
    finally:
        _abi.msf_set_option(_abi.OPT_ROUND_LIMIT, old)


@pytest.mark.parametrize("parts", [1, 7])
@pytest.mark.parametrize("n,m", [(2, 70), (30, 1000000), (63, 2015), (63, 2016), (300, 500000), (300, 2000000),
                                 (2048, 65536), (2048, 65535), (2049, 400000)])
def test_labels_rounds_and_time(n, m, parts):
    from paper_2110_04865_gb300 import api
    rng = np.random.default_rng(n + m)
    s, d = rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32)
    if parts > 1:  # edges inside residue classes only
        d = np.minimum(d - d % parts + s % parts, n - 1)
        d = np.where(d % parts == s % parts, d, s).astype(np.int32)
    g = api.Graph(n, to_dev(s), to_dev(d), to_dev(np.ones(m, np.float32)))
    labels, rounds, t = components(g)
    loop_labels, loop_rounds, loop_t = components(g, 63)
    g.free()
    assert np.array_equal(labels, oracle.kruskal(n, s, d, np.ones(m, np.float32), 0)[1])
    assert np.array_equal(labels, loop_labels) and rounds == loop_rounds
    assert t < loop_t
