"""Zero weights of both signs among others, and alone: equal to the oracle (the
two zeros are one weight), and no slower than another weight shared by all."""
from __future__ import annotations

import time

import numpy as np
import pytest

import oracle
from gpu_util import assert_parity, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_04865_gb300 import build_lib
    build_lib.build()


def ends(n, m):
    rng = np.random.default_rng(n)
    return rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32), rng


@pytest.mark.parametrize("zero", [0.0, 0.1, 0.5, 0.9, 1.0])
@pytest.mark.parametrize("others", ["negative", "positive", "both", "denormal"])
@pytest.mark.parametrize("n,m", [(4096, 100000), (60000, 900000)])
def test_zeros_among_others(n, m, others, zero):
    from paper_2110_04865_gb300 import api
    s, d, rng = ends(n, m)
    w = rng.standard_normal(m).astype(np.float32)
    if others == "denormal":
        w = (rng.integers(-3, 4, m) * 2.0 ** -149).astype(np.float32)
    elif others != "both":
        w = np.abs(w) * (-1 if others == "negative" else 1)
    w = np.where(rng.random(m) < zero, np.where(rng.random(m) < 0.5, np.float32(0.0), np.float32(-0.0)), w)
    w = w.astype(np.float32)
    assert_parity(n, s, d, w, 0)
    copies = np.arange(4, dtype=np.int64)
    got = api.compute_batched(copies * n, copies * m, *(to_dev(np.tile(a, 3)) for a in (s, d, w)))
    ref = oracle.kruskal(n, s, d, w, 0)
    for a, b in zip(got, ref):
        assert np.array_equal(a.cpu().numpy(), np.tile(np.atleast_1d(b), 3))


@pytest.mark.parametrize("n,m", [(4096, 100000), (1 << 20, 1 << 24)])
def test_zeros_take_no_longer_than_ones(n, m):
    import torch
    from paper_2110_04865_gb300 import api
    s, d, _ = ends(n, m)
    arrays = [to_dev(s), to_dev(d)]
    times = []
    for value in (0.0, 1.0):
        w = torch.full((m,), value, device="cuda")
        api.compute(n, *arrays, w)
        ts = []
        for _ in range(7):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            api.compute(n, *arrays, w)
            ts.append(time.perf_counter() - t0)
        times.append(sorted(ts)[3])
    assert times[0] < 1.3 * times[1]
