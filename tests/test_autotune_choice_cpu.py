"""What the autotuner times and sets (no GPU: its timer is a fake that says how
long each call takes under the options of the moment): with the default options
the shape of msf_min_edge's own sweep, and nothing that puts the round loop in
the place of the solvers; with the round loop selected the whole loop."""
from __future__ import annotations

import json

import pytest

torch = pytest.importorskip("torch")

from paper_2110_04865_gb300 import _abi, autotune  # noqa: E402

TUNED = (_abi.OPT_SLOTS_PER_LANE, _abi.OPT_PREFETCH, _abi.OPT_BLOCKS_PER_SM, _abi.OPT_SWEEP, _abi.OPT_COMPACT_TAU)


def setting():
    return tuple(_abi.msf_get_option(o) for o in TUNED)


CPU = torch.device("cpu")


class Graph:
    n, device = 10, CPU

    def stats(self):
        return _abi.Stats(nnz=1 << 20, rows=1 << 16)

    def compute(self, **_):
        pass


@pytest.fixture
def bench(monkeypatch, tmp_path):
    """Records (kind, options) of every timed call; `speed` maps options to ms."""
    from paper_2110_04865_gb300 import build_lib
    build_lib.build()
    calls = []

    class Timer:
        speed = staticmethod(lambda kind, options: 1.0)

        def __init__(self, *_):
            pass

        def call_ms(self, call, reps):
            calls.append(("call", setting()))
            return self.speed("call", setting())

        def sweep_ms(self, graph, parent, reps):
            calls.append(("sweep", setting()))
            return self.speed("sweep", setting())

    monkeypatch.setattr(autotune, "_Timer", Timer)
    monkeypatch.setattr(autotune, "CACHE", str(tmp_path / "autotune.json"))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *_: "a GPU")
    old = {o: _abi.msf_get_option(o) for o in range(15)}
    yield Timer, calls, tmp_path / "autotune.json"
    for o, v in old.items():
        _abi.msf_set_option(o, v)


@pytest.mark.parametrize("objective", ["compute", "sweep"])
def test_default_path_is_left_selected(bench, objective):
    Timer, calls, _ = bench
    # other sweep forms are faster as sweeps, and would bring the loop back
    Timer.speed = staticmethod(lambda kind, o: 0.5 if o[3] else 1.0 if o[:3] == (8, 0, 8) else 2.0)
    best = autotune.tune(Graph(), objective=objective)
    assert {o[3] for _, o in calls} == {0} and {o[4] for _, o in calls} == {0.5}
    assert setting() == (8, 0, 8, 0, 0.5)
    assert [best[k] for k in autotune.CONFIG_KEYS] == [8, 0, 8, 0, 0.5]
    # msf_compute does not depend on the shape: timed once, not per candidate
    assert sum(kind == "call" for kind, _ in calls) == (1 if objective == "compute" else 0)


def test_equal_sweeps_keep_the_default(bench):
    Timer, _, _ = bench
    Timer.speed = staticmethod(lambda kind, o: 1.0 if o[2] == 4 else 0.995)
    autotune.tune(Graph())
    assert setting() == (4, 0, 4, 0, 0.5)


def test_batched_default_path_changes_nothing(bench):
    Timer, calls, _ = bench
    best = autotune.tune_batched(lambda: None, "some batch", device=CPU)
    assert len(calls) == 1 and setting() == (4, 0, 4, 0, 0.5)
    assert best["blocks_per_sm"] == 4 and best["ms"] == 1.0


def test_round_loop_is_tuned_where_it_runs(bench):
    Timer, calls, _ = bench
    Timer.speed = staticmethod(lambda kind, o: 1.0 if (o[:4] == (8, 0, 3, 2) and o[4] == 0.25) else
                               2.0 if o[:4] == (8, 0, 3, 2) else 3.0)
    _abi.msf_set_option(_abi.OPT_BUILD, 1)
    autotune.tune(Graph())
    assert {o[3] for _, o in calls} == {0, 1, 2}
    assert setting() == (8, 0, 3, 2, 0.25)
    calls.clear()
    for o, v in zip(TUNED, (4, 0, 4, 0, 0.5)):
        _abi.msf_set_option(o, v)
    autotune.tune_batched(lambda: None, "some batch", device=CPU)
    assert len(calls) == len(autotune.CANDIDATES) + len(autotune.TAU_CANDIDATES)
    assert setting() == (8, 0, 3, 2, 0.25)


def test_entries_of_an_older_format_are_not_applied(bench):
    _, calls, path = bench
    stale = dict(spl=8, prefetch=0, blocks_per_sm=2, sweep=1, compact_tau=0.0, ms=1.0)
    key = autotune._key(CPU, Graph().stats())
    path.write_text(json.dumps({f"{key}/compute": stale, "a_GPU/batched/some batch": stale}))
    assert not autotune.tune(Graph())["cached"]
    assert not autotune.tune_batched(lambda: None, "some batch", device=CPU)["cached"]
    assert setting()[3:] == (0, 0.5)
    calls.clear()
    assert autotune.tune(Graph())["cached"] and autotune.tune_batched(lambda: None, "some batch", device=CPU)["cached"]
    assert not calls
