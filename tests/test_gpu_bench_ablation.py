"""The bench's ablation of Sec. 4.1 compares two formulations of one thing: both
of its computes are round loops, one with each kernel."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu


def test_both_arms_run_the_round_loop(monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import bench
    from paper_2110_04865_gb300 import _abi, autotune, build_lib
    build_lib.build()
    arms, plain = [], _abi.msf_compute

    def compute(g, *args):
        plain(g, *args)
        st = _abi.msf_get_stats(g)
        arms.append((int(_abi.msf_get_option(_abi.OPT_KERNEL)), autotune.round_loop_selected(), st.rounds,
                     st.forest_edges))

    monkeypatch.setattr(_abi, "msf_compute", compute)
    before = {o: _abi.msf_get_option(o) for o in range(15)}
    dev = torch.device("cuda:0")
    out = bench.bench_pairwise(dev, int(torch.cuda.current_stream(dev).cuda_stream),
                               torch.empty(1 << 20, dtype=torch.uint8, device=dev))
    assert {o: _abi.msf_get_option(o) for o in range(15)} == before
    assert {k for k, *_ in arms} == {0, 1} and all(loop for _, loop, *_ in arms)
    assert len({x[2:] for x in arms}) == 1  # the same rounds and forest
    assert out["same_forest"] and out["compute_speedup"] > 0 and out["sweep_speedup"] > 0
