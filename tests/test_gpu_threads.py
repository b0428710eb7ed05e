"""Calls of several threads, a stream each: every result is the oracle's, and calls
that each fill the device share it."""
from __future__ import annotations

import threading
import time

import numpy as np
import pytest

import oracle
from gpu_util import to_dev

pytestmark = pytest.mark.gpu

T = 8


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


def in_threads(work):
    import torch
    errors = []

    def body(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                work(i)
        except BaseException as e:  # (reported by the test's thread)
            errors.append(e)

    ts = [threading.Thread(target=body, args=(i,)) for i in range(T)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if errors:
        raise errors[0]


def same(got, ref):
    return all(np.array_equal(a.cpu().numpy(), np.atleast_1d(b)) for a, b in zip(got, ref))


def test_mixed_calls():
    import torch
    from paper_2110_04865_gb300 import api
    sizes = [(100, 300), (4096, 32768), (30000, 200000), (70000, 140000), (200000, 1200000), (1 << 18, 1 << 22)]
    graphs = [(n, m) + make(n, m, k) for k, (n, m) in enumerate(sizes)]
    refs = [oracle.kruskal(n, s, d, w, 0) for n, m, s, d, w in graphs]
    dev = [[to_dev(a) for a in g[2:]] for g in graphs]
    voff = np.concatenate([[0], np.cumsum([g[0] for g in graphs[:4]])]).astype(np.int64)
    eoff = np.concatenate([[0], np.cumsum([g[1] for g in graphs[:4]])]).astype(np.int64)
    whole = [torch.cat([x[k] for x in dev[:4]]) for k in range(3)]
    parts = [np.concatenate([np.atleast_1d(r[k]) for r in refs[:4]]) for k in range(3)]
    torch.cuda.synchronize()

    def work(i):
        rng = np.random.default_rng(i)
        for _ in range(12):
            k = int(rng.integers(0, len(sizes)))
            n = sizes[k][0]
            kind = int(rng.integers(0, 3))
            if kind == 0:
                assert same(api.compute(n, *dev[k]), refs[k])
            elif kind == 1:
                g = api.Graph(n, *dev[k])
                assert same(g.compute(), refs[k])
                assert np.array_equal(g.components().cpu().numpy(), refs[k][1])
                g.free()
            else:
                assert same(api.compute_batched(voff, eoff, *whole), parts)

    in_threads(work)


@pytest.mark.parametrize("n,m", [(65536, 1 << 18), (65536, 1 << 20)])
def test_calls_share_the_device(n, m):
    """Eight threads take well under eight times one thread's time (calls that
    each wait for the whole device take nearly that)."""
    import torch
    from paper_2110_04865_gb300 import api
    graphs = [api.Graph(n, *(to_dev(a) for a in make(n, m, i))) for i in range(T)]
    torch.cuda.synchronize()

    def work(i):
        for _ in range(25):
            graphs[i].compute()

    times = []
    for run in (lambda: in_threads(work), lambda: [work(i) for i in range(T)]):
        ts = []
        for _ in range(4):
            t0 = time.perf_counter()
            run()
            torch.cuda.synchronize()
            ts.append(time.perf_counter() - t0)
        times.append(min(ts[1:]))
    for g in graphs:
        g.free()
    assert times[0] < 0.65 * times[1]
