"""msf_compute on a handle solves from the edges the build kept: the forest,
labels, total, forest size and round count are the round loop's over the CSR
(the host-driven loop runs the same steps), with and without the confirming
last round, for both input forms, at the sizes where the routes change."""
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


def check(n, src, dst, w, row_ptr=None):
    from paper_2110_04865_gb300 import _abi, api
    g = api.Graph(n, None if src is None else to_dev(src), to_dev(dst), to_dev(w),
                  None if row_ptr is None else to_dev(row_ptr))
    old = {o: _abi.msf_get_option(o) for o in (_abi.OPT_EXEC_MODE, _abi.OPT_EARLY_STOP)}
    try:
        for stop in (1, 0):
            _abi.msf_set_option(_abi.OPT_EARLY_STOP, stop)
            runs = []
            for host_loop in (1, 0, 0):  # (twice on one handle)
                _abi.msf_set_option(_abi.OPT_EXEC_MODE, host_loop)
                out = [x.cpu().numpy() for x in g.compute()]
                st = g.stats()
                runs.append((out, (st.rounds, st.forest_edges, st.n, st.m, st.nnz, st.rows)))
            for out, st in runs[1:]:
                assert st == runs[0][1]
                for a, b in zip(out, runs[0][0]):
                    assert np.array_equal(a, b)
    finally:
        for o, v in old.items():
            _abi.msf_set_option(o, v)
        g.free()
    return runs[0][0]


@pytest.mark.parametrize("n,m", [(1, 0), (1, 4), (2, 1), (50, 7), (300, 900), (4096, 8192), (4096, 8195), (900, 60000),
                                 (12000, 30000), (20000, 131072), (9000, 262147), (300001, 200000),
                                 (4000, 24576), (4000, 24577), (300000, 3145727), (400000, 3145728), (157286, 1572860), (157287, 1572864), (300000, 4194309), (1900000, 3000001), (2600000, 6300009)])
def test_sizes(n, m):
    rng = np.random.default_rng(n + m)
    s, d = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    for w in (rng.standard_normal(m).astype(np.float32), rng.integers(0, 9, m).astype(np.uint32)):
        got = check(n, s, d, w)
        want = oracle.kruskal(n, s, d, w, 0 if w.dtype == np.float32 else 1)
        for a, b in zip(got[:2], want[:2]):
            assert np.array_equal(a, b)
        assert float(got[2][0]) == want[2]


@pytest.mark.parametrize("shape", ["path up", "path mixed", "two halves", "hub"])
def test_rounds_of_special_shapes(shape):
    n = 70001
    rng = np.random.default_rng(4)
    a = np.arange(n - 1, dtype=np.int32)
    s, d, w = a, a + 1, np.arange(n - 1).astype(np.float32)
    if shape == "path mixed":
        w = rng.permutation(w)
    elif shape == "two halves":  # two components: the last round confirms
        keep = a != n // 2
        s, d, w = s[keep], d[keep], rng.permutation(w)[keep]
    elif shape == "hub":
        m = 400000
        s, d, w = np.zeros(m, np.int32), rng.integers(0, n, m).astype(np.int32), rng.random(m).astype(np.float32)
    check(n, s, d, w)


@pytest.mark.parametrize("n,m", [(60, 200), (5000, 40000), (30000, 900000)])
def test_csr_form(n, m):
    rng = np.random.default_rng(m)
    u, v = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    w = rng.random(m).astype(np.float32)
    keep = u != v
    u, v, w = u[keep], v[keep], w[keep]
    row, col, ww = np.concatenate([u, v]), np.concatenate([v, u]), np.concatenate([w, w])
    o = np.lexsort((col, row))
    rp = np.concatenate([[0], np.cumsum(np.bincount(row, minlength=n))]).astype(np.int64)
    check(n, None, col[o].copy(), ww[o].copy(), rp)
