"""The gradient's arrays off a 16-byte boundary: values at the edges of a warp's
share, and a time near that of aligned arrays."""
from __future__ import annotations

import time

import numpy as np
import pytest

from gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_04865_gb300 import build_lib
    build_lib.build()


def backward(m, eoff, mask, gt, gw):
    from paper_2110_04865_gb300 import _abi
    _abi.msf_weight_backward(m, len(eoff) - 1, eoff.ctypes.data, mask.data_ptr(), gt.data_ptr(), gw.data_ptr())


@pytest.mark.parametrize("mask_off,grad_off", [(1, 0), (0, 1), (5, 3)])
@pytest.mark.parametrize("m", [1, 31, 32, 33, 255, 256, 257, 5000, 70001])
@pytest.mark.parametrize("G", [1, 2, 400])
def test_values(G, m, mask_off, grad_off):
    import torch
    rng = np.random.default_rng(m + G)
    eoff = np.concatenate([[0], np.sort(rng.integers(0, m + 1, G - 1)), [m]]).astype(np.int64)
    mask, gt = (rng.random(m) < 0.4).astype(np.uint8), rng.standard_normal(G)
    mk = to_dev(np.concatenate([np.ones(mask_off, np.uint8), mask, np.ones(9, np.uint8)]))
    gw = torch.full((grad_off + m + 9,), 7.0, device="cuda")
    backward(m, eoff, mk[mask_off:], to_dev(gt), gw[grad_off:])
    graph = np.clip(np.searchsorted(eoff[:G], np.arange(m), side="right") - 1, 0, G - 1)
    got = gw.cpu().numpy()
    assert np.array_equal(got[grad_off:grad_off + m], np.where(mask != 0, gt[graph].astype(np.float32), np.float32(0)))
    assert (got[:grad_off] == 7).all() and (got[grad_off + m:] == 7).all()


@pytest.mark.parametrize("fill", [0, 1])
def test_time(fill):
    import torch
    m, G = 1 << 26, 900
    eoff = np.linspace(0, m, G + 1).astype(np.int64)
    mask = torch.full((m + 16,), fill, dtype=torch.uint8, device="cuda")
    gt, gw = torch.ones(G, dtype=torch.float64, device="cuda"), torch.empty(m + 16, device="cuda")
    times = []
    for off in (0, 1):
        ts = []
        for _ in range(9):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            backward(m, eoff, mask[off:], gt, gw[off:])
            torch.cuda.synchronize()
            ts.append(time.perf_counter() - t0)
        times.append(sorted(ts)[4])
    assert times[1] < 1.7 * times[0]
