"""One graph solved from its edge list (api.compute, msf_compute_batched with
G = 1): bit-exact against the oracle and the CSR round loop at the sizes where
its parts begin and end -- batches of 128 edges, warp and block regions, one
and two light classes, the heavy filter with its bitmap in shared and in global
memory -- and on inputs that stress the thresholds and the parent chains."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gpu_util import DEV, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_04865_gb300 import build_lib
    build_lib.build()


def check(n, s, d, w, csr=True):
    from paper_2110_04865_gb300 import _abi, api
    wtype = 0 if w.dtype == np.float32 else 1
    got = api.compute(n, to_dev(s), to_dev(d), to_dev(w))
    omk, olb, otot = oracle.kruskal(n, s, d, w, wtype)
    assert np.array_equal(got[0].cpu().numpy(), omk)
    assert np.array_equal(got[1].cpu().numpy(), olb)
    assert float(got[2].cpu()[0]) == otot
    if csr:
        old = _abi.msf_get_option(_abi.OPT_BUILD)
        try:
            _abi.msf_set_option(_abi.OPT_BUILD, 1)  # an explicit builder: the round loop over a CSR
            ref = api.compute(n, to_dev(s), to_dev(d), to_dev(w))
        finally:
            _abi.msf_set_option(_abi.OPT_BUILD, old)
        for a, b in zip(got, ref):
            assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())


@pytest.mark.parametrize("wtype", [0, 1])
@pytest.mark.parametrize("n,m", [(1, 0), (1, 5), (2, 1), (127, 128), (129, 127), (8193, 4097), (100, 65535),
                                 (40000, 65536), (65536, 65537), (9000, 262147), (1700000, 300001),
                                 (1900000, 3000001), (500001, 4194304), (2600000, 4300009),
                                 (393215, 4194305), (393216, 4194304), (917503, 1300000), (917504, 1300000)])
def test_sizes(n, m, wtype):
    rng = np.random.default_rng(n + m)
    s = rng.integers(0, n, m).astype(np.int32)
    d = rng.integers(0, n, m).astype(np.int32)
    if m > 9:
        s[:3] = d[:3]                                   # self-loops
        s[-2:], d[-2:] = s[3:5], d[3:5]                 # duplicate edges
    w = rng.standard_normal(m).astype(np.float32) if wtype == 0 else rng.integers(0, 9, m).astype(np.uint32)
    check(n, s, d, w)


@pytest.mark.parametrize("kind", ["zeros", "signed zeros", "inf", "denormal", "max", "ascending", "descending"])
def test_weights_at_the_thresholds(kind):
    """Ties across the thresholds (all weights equal, few values, both zeros),
    infinities, denormals, and weights in the order of the edges."""
    n, m = 30000, 400003
    rng = np.random.default_rng(7)
    s = rng.integers(0, n, m).astype(np.int32)
    d = rng.integers(0, n, m).astype(np.int32)
    w = {"zeros": np.zeros(m, np.float32),
         "signed zeros": rng.choice(np.array([0.0, -0.0, 1.0, -1.0], np.float32), m),
         "inf": rng.choice(np.array([-np.inf, np.inf, 2.0], np.float32), m, p=[0.5, 0.25, 0.25]),
         "denormal": (rng.standard_normal(m) * 1e-40).astype(np.float32),
         "max": np.full(m, 0xFFFFFFFF, np.uint32),
         "ascending": np.sort(rng.random(m).astype(np.float32)),
         "descending": np.sort(rng.random(m).astype(np.float32))[::-1].copy()}[kind]
    if kind == "inf":  # both infinities in one forest have no sum: only the mask and labels are compared
        from paper_2110_04865_gb300 import api
        got = api.compute(n, to_dev(s), to_dev(d), to_dev(w))
        omk, olb, _ = oracle.kruskal(n, s, d, np.nan_to_num(w, posinf=3e38, neginf=-3e38), 0)
        assert np.array_equal(got[0].cpu().numpy(), omk) and np.array_equal(got[1].cpu().numpy(), olb)
        return
    check(n, s, d, w)


@pytest.mark.parametrize("order", ["ascending", "descending", "random"])
def test_long_chains(order):
    """A path whose roots all hook the same way in one round (chains of as many
    hops as there are vertices), and one with random weights."""
    n = 700001
    w = np.arange(n - 1).astype(np.float32)
    if order == "descending":
        w = w[::-1].copy()
    if order == "random":
        w = np.random.default_rng(3).permutation(w)
    a = np.arange(n - 1, dtype=np.int32)
    check(n, a, a + 1, w)


def test_hub_and_many_components():
    rng = np.random.default_rng(11)
    n, m = 50000, 600000
    d = rng.integers(0, n, m).astype(np.int32)
    check(n, np.zeros(m, np.int32), d, rng.random(m).astype(np.float32))
    s = (rng.integers(0, n, m) // 8 * 8).astype(np.int32)
    check(n, s, (s + rng.integers(0, 8, m)).astype(np.int32), rng.random(m).astype(np.float32))


def test_unaligned_host_and_absent_outputs():
    import torch
    from paper_2110_04865_gb300 import _abi, api
    rng = np.random.default_rng(2)
    n, m = 5000, 200001
    s, d = (rng.integers(0, n, m + 1).astype(np.int32) for _ in range(2))
    w = rng.random(m + 1).astype(np.float32)
    omk, olb, otot = oracle.kruskal(n, s[1:].copy(), d[1:].copy(), w[1:].copy(), 0)
    for got in (api.compute(n, to_dev(s)[1:], to_dev(d)[1:], to_dev(w)[1:]),
                api.compute(n, s[1:].copy(), d[1:].copy(), w[1:].copy())):
        got = [x.cpu().numpy() if isinstance(x, torch.Tensor) else x for x in got]
        assert np.array_equal(got[0], omk) and np.array_equal(got[1], olb) and float(got[2][0]) == otot
    off = np.array([0, n, 0, m], np.int64)
    S, D, W = to_dev(s)[1:], to_dev(d)[1:], to_dev(w)[1:]
    mk = torch.empty(m + 3, dtype=torch.uint8, device=DEV)[3:]
    for outs in ((mk.data_ptr(), 0, 0), (0, 0, 0)):
        _abi.msf_compute_batched(1, off.ctypes.data, off.ctypes.data + 16, S.data_ptr(), D.data_ptr(), W.data_ptr(),
                                 0, *outs)
    assert np.array_equal(mk.cpu().numpy(), omk)


@pytest.mark.parametrize("m", [300, 400000])
def test_invalid_edges_are_refused(m):
    from paper_2110_04865_gb300 import _abi, api
    rng = np.random.default_rng(m)
    n = 200
    for what, message in (("high", "index"), ("negative", "index"), ("nan", "NaN")):
        s, d = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
        w = rng.random(m).astype(np.float32)
        if what == "high":
            s[m // 2] = n
        elif what == "negative":
            d[m - 1] = -1
        else:
            w[m // 3] = np.nan
        with pytest.raises(_abi.MsfError, match=message) as e:
            api.compute(n, to_dev(s), to_dev(d), to_dev(w))
        assert e.value.code == 1
    check(n, *(rng.integers(0, n, m).astype(np.int32) for _ in range(2)), rng.random(m).astype(np.float32))
