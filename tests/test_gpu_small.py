"""Graphs solved one block each in shared memory (msf_compute_batched when all
of them fit, api.compute on a small graph): bit-exact against the oracle and
the CSR round loop at the sizes where the path's parts begin and end -- edges
kept in registers (8 per thread of 256, 512 or 1024), lists, the filter, the
largest graph that fits -- with empty graphs, ties and invalid edges."""
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


def make(rng, nv, ne, wtype):
    nv, ne = np.asarray(nv, np.int64), np.asarray(ne, np.int64)
    voff, eoff = (np.concatenate([[0], np.cumsum(x)]).astype(np.int64) for x in (nv, ne))
    lim = np.repeat(nv, ne)
    m = len(lim)
    s, d = ((rng.random(m) * lim).astype(np.int32) for _ in range(2))
    w = rng.standard_normal(m).astype(np.float32) if wtype == 0 else rng.integers(0, 6, m).astype(np.uint32)
    return voff, eoff, s, d, w


def check(voff, eoff, s, d, w):
    from paper_2110_04865_gb300 import _abi, api
    wtype = 0 if w.dtype == np.float32 else 1
    got = api.compute_batched(voff, eoff, to_dev(s), to_dev(d), to_dev(w))
    ref = oracle.kruskal_batched(voff, eoff, s, d, w, wtype)
    for a, b in zip(got, ref):
        assert np.array_equal(a.cpu().numpy(), b)
    old = _abi.msf_get_option(_abi.OPT_BUILD)
    try:
        _abi.msf_set_option(_abi.OPT_BUILD, 1)  # an explicit builder: the round loop over a CSR
        csr = api.compute_batched(voff, eoff, to_dev(s), to_dev(d), to_dev(w))
    finally:
        _abi.msf_set_option(_abi.OPT_BUILD, old)
    for a, b in zip(got, csr):
        assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())


@pytest.mark.parametrize("wtype", [0, 1])
@pytest.mark.parametrize("n,m", [(1, 0), (1, 3), (2, 1), (33, 31), (300, 512), (300, 513), (2000, 8191), (2000, 8192),
                                 (2000, 8193), (900, 40001), (60, 70000), (16000, 16001), (19000, 70003),
                                 (20500, 9000)])
def test_one_graph(n, m, wtype):
    check(*make(np.random.default_rng(n + m), [n], [m], wtype))


@pytest.mark.parametrize("wtype", [0, 1])
@pytest.mark.parametrize("G,nmax,deg", [(3, 40, 4), (40, 3000, 12), (152, 500, 3), (153, 500, 3), (400, 60, 30),
                                        (200, 9000, 4)])
def test_batches(G, nmax, deg, wtype):
    """Fewer graphs than SMs (one block size) and more (three, side by side);
    empty graphs and graphs without edges among them."""
    rng = np.random.default_rng(G + nmax)
    nv = rng.integers(0, nmax, G)
    nv[1], nv[2 % G] = 0, nmax
    ne = np.where(nv > 0, rng.integers(0, nmax * deg, G), 0)
    ne[2 % G] = nmax * deg
    if G > 5:
        ne[5] = 0
    check(*make(rng, nv, ne, wtype))


@pytest.mark.parametrize("kind", ["equal", "ascending", "descending", "path"])
def test_ties_orders_and_chains(kind):
    rng = np.random.default_rng(5)
    n, m = 6000, 50000
    voff, eoff, s, d, _ = make(rng, [n], [m], 0)
    if kind == "path":
        s, d = np.arange(n - 1, dtype=np.int32), np.arange(1, n, dtype=np.int32)
        eoff = np.array([0, n - 1], np.int64)
    w = np.arange(len(s)).astype(np.float32)
    w = {"equal": np.full(len(s), 2.5, np.float32), "ascending": w, "descending": w[::-1].copy(), "path": w}[kind]
    check(voff, eoff, s, d, w)


def test_unaligned_edges_and_host_arrays():
    import torch
    from paper_2110_04865_gb300 import api
    rng = np.random.default_rng(8)
    voff, eoff, s, d, w = make(rng, [700, 900, 1300], [1001, 20003, 9999], 0)
    ref = oracle.kruskal_batched(voff, eoff, s, d, w, 0)
    pad = [to_dev(np.concatenate([a[:1], a])) for a in (s, d, w)]
    for got in (api.compute_batched(voff, eoff, *(a[1:] for a in pad)), api.compute_batched(voff, eoff, s, d, w)):
        for a, b in zip(got, ref):
            assert np.array_equal(a.cpu().numpy() if isinstance(a, torch.Tensor) else a, b)


@pytest.mark.parametrize("what", ["high", "negative", "nan", "no vertices"])
@pytest.mark.parametrize("G", [1, 200])
def test_invalid_edges_are_refused(G, what):
    """An index outside its own graph (inside the batch) is invalid too."""
    from paper_2110_04865_gb300 import _abi, api
    rng = np.random.default_rng(G)
    voff, eoff, s, d, w = make(rng, [50] * G, [2000] * G, 0)
    at = (G // 2) * 2000 + 17
    if what == "high":
        s[at] = 50
    elif what == "negative":
        d[at] = -1
    elif what == "nan":
        w[at] = np.nan
    else:
        voff = np.maximum(voff - 50, 0)  # the first graph has edges and no vertices
    with pytest.raises(_abi.MsfError) as e:
        api.compute_batched(voff, eoff, to_dev(s), to_dev(d), to_dev(w))
    assert e.value.code == 1
