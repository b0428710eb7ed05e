"""Batches with graphs that do not fit in one thread block: the larger ones are
solved together from their edge lists, next to the small ones.  Bit-exact
against the oracle and the union round loop over shapes that meet the pages,
the graph boundaries inside them and the block solver's limits."""
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


SHAPES = {
    "empty and large": ([0, 70000, 5, 0, 25000, 1, 40000, 0], [0, 600001, 9, 0, 3, 2, 77, 0]),
    "limits of a block": ([21000, 21400, 21600, 65536, 65537, 128, 3], [524288, 524289, 131, 127, 129, 600000, 0]),
    "two large": ([300001, 299999], [1700003, 2600007]),
    "odd starts": ([30000 + 7 * i for i in range(24)], [20001 + 1777 * i for i in range(24)]),
    "mixed": ([64 + 911 * i for i in range(60)], [16 + 4001 * i for i in range(60)]),
}


def batch(shape, kind):
    nv, ne = (np.array(x, np.int64) for x in SHAPES[shape])
    rng = np.random.default_rng(len(nv))
    voff, eoff = (np.concatenate([[0], np.cumsum(x)]).astype(np.int64) for x in (nv, ne))
    lim, m = np.repeat(nv, ne), int(eoff[-1])
    s, d = ((rng.random(m) * lim).astype(np.int32) for _ in range(2))
    if kind == "u32":
        w = rng.integers(0, 5, m).astype(np.uint32)
    else:
        w = rng.standard_normal(m).astype(np.float32)
        if kind == "scales":  # every graph with weights of its own magnitude
            w *= np.repeat(10.0 ** rng.integers(-30, 30, len(nv)), ne).astype(np.float32)
    return voff, eoff, s, d, w


@pytest.mark.parametrize("kind", ["f32", "u32", "scales"])
@pytest.mark.parametrize("shape", SHAPES)
def test_batch_equals_oracle_and_round_loop(shape, kind):
    from paper_2110_04865_gb300 import _abi, api
    voff, eoff, s, d, w = batch(shape, kind)
    want = oracle.kruskal_batched(voff, eoff, s, d, w, 1 if kind == "u32" else 0)
    # device arrays that start off a 16-byte boundary too
    S, D, W = (to_dev(np.concatenate([x[:1], x])) if shape == "odd starts" else to_dev(x) for x in (s, d, w))
    if shape == "odd starts":
        S, D, W = S[1:], D[1:], W[1:]
    got = api.compute_batched(voff, eoff, S, D, W)
    old = _abi.msf_get_option(_abi.OPT_BUILD)
    try:
        _abi.msf_set_option(_abi.OPT_BUILD, 1)  # an explicit builder: the round loop over the union's CSR
        ref = api.compute_batched(voff, eoff, S, D, W)
    finally:
        _abi.msf_set_option(_abi.OPT_BUILD, old)
    for a, b, c in zip(got, ref, want):
        assert np.array_equal(a.cpu().numpy(), c) and np.array_equal(b.cpu().numpy(), c)


@pytest.mark.parametrize("what", ["high", "negative", "nan"])
def test_invalid_edge_in_a_large_graph(what):
    from paper_2110_04865_gb300 import _abi, api
    voff, eoff, s, d, w = batch("odd starts", "f32")
    at = int(eoff[-2]) + 5
    if what == "high":
        s[at] = voff[-1] - voff[-2]
    elif what == "negative":
        d[at] = -1
    else:
        w[at] = np.nan
    with pytest.raises(_abi.MsfError, match="NaN" if what == "nan" else "index") as e:
        api.compute_batched(voff, eoff, to_dev(s), to_dev(d), to_dev(w))
    assert e.value.code == 1
