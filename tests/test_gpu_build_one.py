"""The one-block build of a small graph: the loop over its CSR, msf_min_edge and
the statistics agree with the oracle and with the multi-launch builder at the
block's limits, for both input forms; bad input is refused."""
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


def graph(n, m, csr, seed=0):
    rng = np.random.default_rng(n + m + seed)
    s, d = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    w = rng.integers(0, 40, m).astype(np.uint32)
    if not csr:
        return s, d, w, None
    rp = np.concatenate([[0], np.cumsum(np.bincount(s, minlength=n))]).astype(np.int64)
    row = np.sort(s)
    return np.where(row < d, row, d).astype(np.int32), d, w, rp


@pytest.mark.parametrize("csr", [False, True])
@pytest.mark.parametrize("n,m", [(1, 0), (1, 9), (2, 1), (7, 5), (1023, 300), (1025, 2047), (8192, 12288),
                                 (8192, 12289), (8192, 16384), (8192, 16385), (8193, 16384), (3, 16384), (8000, 700)])
def test_same_graph(n, m, csr):
    from paper_2110_04865_gb300 import _abi, api
    s, d, w, rp = graph(n, m, csr)
    want = oracle.kruskal(n, s, d, w, 1)
    p = np.arange(n, dtype=np.int32) // 3 * 3
    seen = []
    old = {o: _abi.msf_get_option(o) for o in (_abi.OPT_BUILD, _abi.OPT_EXEC_MODE)}
    try:
        for mode in (0, 1):
            _abi.msf_set_option(_abi.OPT_BUILD, mode)
            g = api.Graph(n, None if csr else to_dev(s), to_dev(d), to_dev(w), None if rp is None else to_dev(rp))
            _abi.msf_set_option(_abi.OPT_EXEC_MODE, 1)  # the loop over the CSR
            got = [x.cpu().numpy() for x in g.compute()]
            _abi.msf_set_option(_abi.OPT_EXEC_MODE, 0)
            st = g.stats()
            seen.append((g.min_edge(to_dev(p)).cpu().numpy(), g.components().cpu().numpy(), st.nnz, st.rows, st.builder))
            g.free()
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]) and float(got[2][0]) == want[2]
    finally:
        for o, v in old.items():
            _abi.msf_set_option(o, v)
    for a, b in zip(*seen):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("csr", [False, True])
@pytest.mark.parametrize("what,message", [("high", "index"), ("negative", "index"), ("nan", "NaN"), ("rows", "row_ptr")])
def test_refused(what, message, csr):
    from paper_2110_04865_gb300 import _abi, api
    if what == "rows" and not csr:
        return
    n, m = 50, 400
    s, d, _, rp = graph(n, m, csr)
    w = np.ones(m, np.float32)
    if what == "high":
        d[m // 2] = n
    elif what == "negative":
        d[m - 1] = -1
    elif what == "nan":
        w[3] = np.nan
    else:
        rp[20] = rp[21] + 1
    with pytest.raises(_abi.MsfError, match=message) as e:
        api.Graph(n, None if csr else to_dev(s), to_dev(d), to_dev(w), None if rp is None else to_dev(rp))
    assert e.value.code == 1
