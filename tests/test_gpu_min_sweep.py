"""msf_min_edge's own sweep (a row's smallest slot tried first) against the
loop's pipelined register sweep (form 2 of MSF_OPT_SWEEP): parents from all roots
to one tree, so that tiles are passed at the first try, slot by slot and in
turn, at the edges of tiles and parts; a refused call leaves r alone."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import DEV, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_04865_gb300 import build_lib
    build_lib.build()


def parents(n, rng):
    yield np.arange(n)
    for k in (max(1, n // 7), max(1, n // 100), min(n, 3), 1):
        p = rng.integers(0, k, n)
        p[:k] = np.arange(k)
        yield p
    p = np.arange(n)  # half of the ids in one tree
    p[n // 2:] = n // 2
    yield p


@pytest.mark.parametrize("spl", [4, 8, 16])
@pytest.mark.parametrize("n,m", [(1, 0), (2, 1), (40, 64), (40, 65), (300, 256), (7, 5000), (5000, 4000), (30000, 200003)])
def test_same_minima(n, m, spl):
    import torch
    from paper_2110_04865_gb300 import _abi, api
    rng = np.random.default_rng(n + m)
    s, d = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    if m > 1000:
        s[: m // 3] = 0  # a row over many tiles
    g = api.Graph(n, to_dev(s), to_dev(d), to_dev(rng.integers(0, 50, m).astype(np.uint32)))
    old = {o: _abi.msf_get_option(o) for o in (_abi.OPT_SWEEP, _abi.OPT_SLOTS_PER_LANE)}
    try:
        _abi.msf_set_option(_abi.OPT_SLOTS_PER_LANE, spl)
        for p in parents(n, rng):
            pt = to_dev(p.astype(np.int32))
            _abi.msf_set_option(_abi.OPT_SWEEP, 2)
            ref = g.min_edge(pt)
            _abi.msf_set_option(_abi.OPT_SWEEP, 0)
            assert torch.equal(g.min_edge(pt), ref)
            acc = torch.full((n,), -1, dtype=torch.int64, device=DEV).cpu().numpy().view(np.uint64)
            for k in range(3):
                r = torch.empty(n, dtype=torch.int64, device=DEV)
                _abi.msf_min_edge_part(g.handle, pt.data_ptr(), k, 3, r.data_ptr())
                acc = np.minimum(acc, r.cpu().numpy().view(np.uint64))
            assert np.array_equal(acc, ref.cpu().numpy().view(np.uint64))
    finally:
        for o, v in old.items():
            _abi.msf_set_option(o, v)
        g.free()


@pytest.mark.parametrize("value", [-1, 50])
def test_refused_parents_leave_r(value):
    import torch
    from paper_2110_04865_gb300 import _abi, api
    rng = np.random.default_rng(1)
    s, d = (rng.integers(0, 50, 400).astype(np.int32) for _ in range(2))
    g = api.Graph(50, to_dev(s), to_dev(d), to_dev(rng.random(400).astype(np.float32)))
    p = np.arange(50, dtype=np.int32)
    p[33] = value
    pt, r = to_dev(p), torch.full((50,), 7, dtype=torch.int64, device=DEV)
    for call in (lambda: _abi.msf_min_edge(g.handle, pt.data_ptr(), r.data_ptr()),
                 lambda: _abi.msf_min_edge_part(g.handle, pt.data_ptr(), 0, 2, r.data_ptr())):
        with pytest.raises(_abi.MsfError, match="parent") as e:
            call()
        assert e.value.code == 1
        torch.cuda.synchronize()
        assert bool((r == 7).all())
    g.free()
