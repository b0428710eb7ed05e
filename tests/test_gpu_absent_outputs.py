"""Any output of a call may be absent: the others are those of the full call,
for every combination, on graphs of each of the solvers' kinds."""
from __future__ import annotations

import itertools

import numpy as np
import pytest

import oracle
from gpu_util import to_dev

pytestmark = pytest.mark.gpu

COMBINATIONS = list(itertools.product((True, False), repeat=3))


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_04865_gb300 import build_lib
    build_lib.build()


def make(nv, ne, wtype, seed=11):
    nv, ne = np.asarray(nv, np.int64), np.asarray(ne, np.int64)
    rng = np.random.default_rng(seed)
    voff, eoff = (np.concatenate([[0], np.cumsum(x)]).astype(np.int64) for x in (nv, ne))
    m, lim = int(eoff[-1]), np.repeat(nv, ne)
    s, d = ((rng.random(m) * lim).astype(np.int32) for _ in range(2))
    w = rng.standard_normal(m).astype(np.float32) if wtype == 0 else rng.integers(0, 9, m).astype(np.uint32)
    return voff, eoff, s, d, w


def call(voff, eoff, arrays, wtype, want):
    """msf_compute_batched with the outputs of `want`; the outputs as arrays
    (None for an absent one), filled with what no result is before."""
    import torch
    from paper_2110_04865_gb300 import _abi
    outs = [torch.full((int(k),), 77, dtype=t, device="cuda") if on else None
            for on, k, t in zip(want, (eoff[-1], voff[-1], len(voff) - 1), (torch.uint8, torch.int32, torch.float64))]
    _abi.msf_compute_batched(len(voff) - 1, voff.ctypes.data, eoff.ctypes.data, *(a.data_ptr() for a in arrays), wtype,
                             *(o.data_ptr() if o is not None else 0 for o in outs),
                             int(torch.cuda.current_stream().cuda_stream))
    return [None if o is None else o.cpu().numpy() for o in outs]


@pytest.mark.parametrize("wtype", [0, 1])
@pytest.mark.parametrize("nv,ne", [([70000, 90001], [300001, 150007]), ([300, 70000, 0, 5000], [900, 40000, 0, 60001])])
def test_batch_with_large_graphs(nv, ne, wtype):
    voff, eoff, s, d, w = make(nv, ne, wtype)
    ref = oracle.kruskal_batched(voff, eoff, s, d, w, wtype)
    arrays = [to_dev(a) for a in (s, d, w)]
    for want in COMBINATIONS:
        for got, r in zip(call(voff, eoff, arrays, wtype, want), ref):
            assert got is None or np.array_equal(got, r), want


@pytest.mark.parametrize("wtype", [0, 1])
@pytest.mark.parametrize("nv,ne", [([40], [512]), ([1500], [8192]), ([700], [30000]),
                                   ([1500] * 40, [8192] * 40), ([60] * 400, [2048] * 400)])
def test_small_graphs(nv, ne, wtype):
    """Blocks of 256, 512 and 1024 threads, the last warp of each holding
    edges (the sizes are those at which every register place is used)."""
    voff, eoff, s, d, w = make(nv, ne, wtype)
    ref = oracle.kruskal_batched(voff, eoff, s, d, w, wtype)
    arrays = [to_dev(a) for a in (s, d, w)]
    for want in COMBINATIONS * 4:
        for got, r in zip(call(voff, eoff, arrays, wtype, want), ref):
            assert got is None or np.array_equal(got, r), want


@pytest.mark.parametrize("n,m", [(50, 200), (1500, 8192), (1500, 24576), (30000, 120000), (300000, 3500000)])
def test_kept_graph(n, m):
    import torch
    from paper_2110_04865_gb300 import _abi, api
    voff, eoff, s, d, w = make([n], [m], 0)
    ref = oracle.kruskal(n, s, d, w, 0)
    g = api.Graph(n, *(to_dev(a) for a in (s, d, w)))
    for want in COMBINATIONS:
        outs = [torch.full((k,), 77, dtype=t, device="cuda") if on else None
                for on, k, t in zip(want, (m, n, 1), (torch.uint8, torch.int32, torch.float64))]
        _abi.msf_compute(g.handle, *(o.data_ptr() if o is not None else 0 for o in outs),
                         int(torch.cuda.current_stream().cuda_stream))
        for o, r in zip(outs, ref):
            assert o is None or np.array_equal(o.cpu().numpy(), np.atleast_1d(r)), want
    g.free()
