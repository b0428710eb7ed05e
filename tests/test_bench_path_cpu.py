"""The bench names what ran: the path of msf_compute and the bytes of the sweep
follow the options (no GPU)."""
from __future__ import annotations

import pytest

pytest.importorskip("torch")


@pytest.fixture
def options():
    from paper_2110_04865_gb300 import _abi, build_lib
    build_lib.build()
    old = {o: _abi.msf_get_option(o) for o in range(15)}
    yield _abi
    for o, v in old.items():
        _abi.msf_set_option(o, v)


def test_defaults(options):
    import bench
    assert bench.sweep_and_path() == (12, "edges")


@pytest.mark.parametrize("option,value,want", [
    ("OPT_SWEEP", 2, (16, "loop")), ("OPT_KERNEL", 1, (16, "loop")), ("OPT_EXEC_MODE", 1, (12, "loop")),
    ("OPT_COMPACT_TAU", 0.25, (12, "loop")), ("OPT_BUILD", 1, (12, "loop")), ("OPT_SHORTCUT", 1, (12, "loop")),
    ("OPT_ROUND_LIMIT", 10, (12, "loop")), ("OPT_SLOTS_PER_LANE", 8, (12, "edges")),
    ("OPT_BLOCKS_PER_SM", 2, (12, "edges"))])
def test_options(options, option, value, want):
    import bench
    options.msf_set_option(getattr(options, option), value)
    assert bench.sweep_and_path() == want
