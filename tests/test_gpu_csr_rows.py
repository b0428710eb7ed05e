"""CSR input: the rows of the slots at the edges of a lane's and a warp's share,
long and empty rows, and the builder for scattered columns, against the oracle
on the slots with row < column; bad rows, columns and weights are refused."""
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


def slots(kind):
    """(row_ptr, columns): any columns, any order, lower triangle ignored."""
    rng = np.random.default_rng(8)
    if kind == "one":
        deg = np.array([3])
    elif kind == "short":
        deg = np.array([0, 0, 1, 15, 0, 16, 17, 0])
    elif kind == "warp":
        deg = np.concatenate([np.full(31, 16), [17], np.zeros(40, int), [511, 513, 0, 1025]])
    elif kind == "empty ends":
        deg = np.concatenate([np.zeros(3000, int), rng.integers(0, 9, 2000), np.zeros(3001, int)])
    elif kind == "long":
        deg = np.concatenate([[200001], rng.integers(0, 40, 9000), [70000]])
    else:  # scattered
        deg = rng.integers(0, 121, 215000)  # 12.9 M slots: the bucketed builder
    n = len(deg)
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    return rp, rng.integers(0, n, int(rp[-1])).astype(np.int32)


@pytest.mark.parametrize("kind", ["one", "short", "warp", "empty ends", "long", "scattered"])
def test_rows(kind):
    from paper_2110_04865_gb300 import _abi, api
    rp, col = slots(kind)
    n, m = len(rp) - 1, len(col)
    w = np.random.default_rng(1).random(m).astype(np.float32)
    row = np.repeat(np.arange(n), np.diff(rp)).astype(np.int32)
    want = oracle.kruskal(n, np.where(row < col, row, col), col, w, 0)
    g = api.Graph(n, None, to_dev(col), to_dev(w), to_dev(rp))
    got = [x.cpu().numpy() for x in g.compute()]
    key, old = _abi.OPT_EXEC_MODE, _abi.msf_get_option(_abi.OPT_EXEC_MODE)
    try:
        _abi.msf_set_option(key, 1)  # the loop over the slots that were built
        loop = [x.cpu().numpy() for x in g.compute()]
    finally:
        _abi.msf_set_option(key, old)
        builder = g.stats().builder
        g.free()
    for a in (got, loop):
        assert np.array_equal(a[0], want[0]) and np.array_equal(a[1], want[1]) and float(a[2][0]) == want[2]
    assert builder == (3 if kind == "scattered" else 1)


@pytest.mark.parametrize("kind", ["long", "scattered"])
@pytest.mark.parametrize("what,message", [("column", "index"), ("negative", "index"), ("rows", "row_ptr"), ("nan", "NaN")])
def test_refused(kind, what, message):
    from paper_2110_04865_gb300 import _abi, api
    rp, col = slots(kind)
    n, m = len(rp) - 1, len(col)
    w = np.ones(m, np.float32)
    if what == "column":
        col[m // 2] = n
    elif what == "negative":
        col[m - 1] = -3
    elif what == "nan":  # (in an ignored slot too)
        col[-1], w[-1] = 0, np.nan
    else:
        rp[n // 2] = rp[n // 2 + 1] + 1
    with pytest.raises(_abi.MsfError, match=message) as e:
        api.Graph(n, None, to_dev(col), to_dev(w), to_dev(rp))
    assert e.value.code == 1
