"""msf_weight_backward with the offsets in the launch's parameters (few graphs)
and with a copy of them (more): the gradient by definition, at the edges of the
16-edge words, with empty graphs, unaligned buffers and offsets that end early."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import DEV, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_04865_gb300 import build_lib
    build_lib.build()


@pytest.mark.parametrize("shift", [0, 3])
@pytest.mark.parametrize("G,m", [(1, 1), (1, 16), (1, 100003), (2, 15), (3, 17), (70, 4099), (959, 50001), (960, 700000),
                                 (961, 50001), (3000, 70001)])
def test_gradient(G, m, shift):
    import torch
    from paper_2110_04865_gb300 import _abi
    rng = np.random.default_rng(G + m)
    eoff = np.sort(rng.integers(0, m + 1, G + 1)).astype(np.int64)
    eoff[0], eoff[-1] = 0, m
    if G > 3:
        eoff[1] = 0                      # an empty graph first and one inside
        eoff[3] = eoff[2]
    mask = (rng.random(m) < 0.3).astype(np.uint8)
    gt = rng.standard_normal(G)
    mk = to_dev(np.concatenate([np.zeros(shift, np.uint8), mask]))[shift:]
    for ends in (eoff, np.minimum(eoff, m - m // 5)):  # offsets that end early: the rest is the last graph's
        gw = torch.full((m + shift,), 7.0, dtype=torch.float32, device=DEV)[shift:]
        _abi.msf_weight_backward(m, G, ends.ctypes.data, mk.data_ptr(), to_dev(gt).data_ptr(), gw.data_ptr())
        torch.cuda.synchronize()
        graph = np.clip(np.searchsorted(ends[:G], np.arange(m), side="right") - 1, 0, G - 1)
        assert np.array_equal(gw.cpu().numpy(), np.where(mask != 0, gt[graph].astype(np.float32), np.float32(0)))
