"""Calls that are refused on the host: the library's error, whatever the size
asked for (no GPU needed, the refusal comes before any of its calls)."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2110_04865_gb300 import build_lib
    build_lib.build()


@pytest.mark.parametrize("tensors", [False, True])
@pytest.mark.parametrize("n,code", [(-1, 1), (-(1 << 40), 1), (-(1 << 70), 1), (0, 1), (1 << 31, 6), (1 << 45, 6),
                                    (1 << 70, 6), ((1 << 64) + 5, 6)])
def test_vertex_count_of_one_graph(monkeypatch, n, code, tensors):
    from paper_2110_04865_gb300 import _abi, api
    monkeypatch.setattr(api, "_stream_handle", lambda device: 0)
    arrays = [np.zeros(3, np.int32), np.zeros(3, np.int32), np.zeros(3, np.float32)]
    if tensors:
        arrays = [torch.from_numpy(a) for a in arrays]
    with pytest.raises(_abi.MsfError) as e:
        api.compute(n, *arrays)
    assert e.value.code == code
    if tensors:
        with pytest.raises(_abi.MsfError) as e:
            api.msf_weight(arrays[2], api.Batch([0, n], [0, 3], arrays[0], arrays[1]))
        assert e.value.code == code
