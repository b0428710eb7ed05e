"""The round loop over the CSRs that the automatic builder makes (default calls
solve a kept graph from its edges and do not read its CSR): the loop's forest,
round count with and without the confirming round, and its bound, against the
solvers and the oracle.  A threshold of its own selects the loop."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def options():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_04865_gb300 import _abi, build_lib
    build_lib.build()
    old = {o: _abi.msf_get_option(o) for o in range(15)}
    yield _abi
    for o, v in old.items():
        _abi.msf_set_option(o, v)


def compare(_abi, g, n, want):
    """Solvers and loop on one graph; the loop's statistics."""
    solved, rounds = g.compute(), {}
    for early in (0, 1):
        _abi.msf_set_option(_abi.OPT_EARLY_STOP, early)
        _abi.msf_set_option(_abi.OPT_COMPACT_TAU, 0.5)
        got = g.compute()
        fast = g.stats()
        _abi.msf_set_option(_abi.OPT_COMPACT_TAU, 0.25)
        loop = g.compute()
        st = g.stats()
        assert (st.rounds, st.forest_edges) == (fast.rounds, fast.forest_edges)
        assert st.kernels > fast.kernels
        rounds[early] = st.rounds
        for x in (solved, got, loop):
            for a, b in zip(x, want):
                assert np.array_equal(a.cpu().numpy(), np.atleast_1d(b))
    assert rounds[1] <= rounds[0] <= rounds[1] + 1
    assert 1 <= rounds[0] <= int(np.ceil(np.log2(n))) + 2
    return st


@pytest.mark.parametrize("workload,builder", [("er4096", 1), ("grid64", 1), ("rmat20", 3), ("rmat20p", 3),
                                              ("grid128", 1)])
def test_edge_lists(options, workload, builder):
    from paper_2110_04865_gb300 import api
    d = synth.workload(workload)
    g = api.Graph(d["n"], to_dev(d["src"]), to_dev(d["dst"]), to_dev(d["w"]))
    assert g.stats().builder == builder
    st = compare(options, g, d["n"], oracle.kruskal(d["n"], d["src"], d["dst"], d["w"], d["wtype"]))
    g.free()
    if workload.startswith("grid"):
        assert st.forest_edges == d["n"] - 1


@pytest.mark.parametrize("n,m", [(300, 1500), (3000, 12000), (1 << 18, 7 << 20)])
def test_csr_input(options, n, m):
    """Up to a size at which CSR input is bucketed; arbitrary order inside a row."""
    from paper_2110_04865_gb300 import api
    rng = np.random.default_rng(m)
    u, v = rng.integers(0, n, m), rng.integers(0, n, m)
    u, v = u[u != v], v[u != v]
    w = rng.integers(1, 200, len(u)).astype(np.float32)
    rows, cols, ww = np.concatenate([u, v]), np.concatenate([v, u]), np.concatenate([w, w])
    order = np.argsort(rows, kind="stable")
    rows, cols, ww = rows[order], cols[order].astype(np.int32), ww[order]
    row_ptr = np.searchsorted(rows, np.arange(n + 1)).astype(np.int64)
    g = api.Graph(n, None, to_dev(cols), to_dev(ww), row_ptr=to_dev(row_ptr))
    assert g.stats().builder == (3 if len(cols) >= 12 << 20 else 1)
    compare(options, g, n, oracle.kruskal(n, np.where(rows < cols, rows, cols).astype(np.int32), cols, ww, 0))
    g.free()
