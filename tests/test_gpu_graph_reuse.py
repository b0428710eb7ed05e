"""The round loop's captured graphs are kept by the options that shaped them: the
loop under any two settings after one another runs each setting's own kernels."""
from __future__ import annotations

import itertools

import numpy as np
import pytest

import oracle
import synth
from gpu_util import to_dev

pytestmark = pytest.mark.gpu

# (kernel, sweep form, slots per lane, prefetch)
SETTINGS = [(0, 0, 4, 0), (1, 0, 4, 0), (0, 2, 4, 0), (0, 1, 4, 0), (1, 2, 4, 0), (0, 0, 4, 1), (0, 0, 8, 0)]


@pytest.fixture
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


def test_settings_in_turn(options):
    """(The pairwise kernel reads an array that only its own setting has: its
    graph under another one would read nothing at all.)"""
    from paper_2110_04865_gb300 import api
    d = synth.workload("er4096")
    want = oracle.kruskal(d["n"], d["src"], d["dst"], d["w"], d["wtype"])
    arrays = [to_dev(d[k]) for k in ("src", "dst", "w")]
    options.msf_set_option(options.OPT_COMPACT_TAU, 0.25)  # a threshold of its own: the loop, also on a kept graph
    options.msf_set_option(options.OPT_BUILD, 1)
    for pair in itertools.permutations(SETTINGS, 2):
        for kernel, sweep, spl, prefetch in pair:
            for o, v in ((options.OPT_KERNEL, kernel), (options.OPT_SWEEP, sweep),
                         (options.OPT_SLOTS_PER_LANE, spl), (options.OPT_PREFETCH, prefetch)):
                options.msf_set_option(o, v)
            g = api.Graph(d["n"], *arrays)
            for a, b in zip(g.compute(), want):
                assert np.array_equal(a.cpu().numpy(), np.atleast_1d(b)), pair
            g.free()
