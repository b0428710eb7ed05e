"""The library's host code against a CUDA runtime that executes nothing
(fake_runtime.cpp): what a call queues and gives back, in success and when one
of its allocations or calls fails.  No GPU needed."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SCENARIOS = ["build_one", "build", "build_sampled", "build_csr", "build_csr_large", "build_radix", "build_bucket",
             "compute_small", "compute", "compute_loop", "components", "min_edge", "one_small", "one", "batch_small",
             "batch", "backward"]


@pytest.fixture(scope="session")
def program(tmp_path_factory):
    from paper_2110_04865_gb300 import build_lib
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    build_lib.build()
    out = tmp_path_factory.mktemp("fake")
    include = os.path.join(os.path.dirname(os.path.dirname(build_lib.nvcc())), "include")
    obj, exe = str(out / "fake.o"), str(out / "fake")
    subprocess.run([cxx, "-O1", "-std=c++17", "-w", "-I", os.path.join(build_lib.ROOT, "include"), "-I", build_lib.CSRC,
                    "-I", include, "-c", os.path.join(HERE, "fake_runtime.cpp"), "-o", obj], check=True)
    objs = [o for o in glob.glob(os.path.join(build_lib.OUT, "*.o")) if os.path.basename(o) != "pool.o"]
    subprocess.run([cxx, obj] + objs + ["-o", exe], check=True)
    return exe


def run(program, scenario, *more):
    r = subprocess.run([program, scenario, *more], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    return r.stdout.splitlines()


@pytest.mark.parametrize("scenario", SCENARIOS)
def test_copies_name_their_memory(program, scenario):
    """Page-locked arrays that are read in place are host memory: no copy of
    them is one between device buffers."""
    assert not [x for x in run(program, scenario + " locked") if x.startswith("plain") and "a copy" in x]


@pytest.mark.parametrize("where", ["", " host", " locked"])
@pytest.mark.parametrize("scenario", SCENARIOS)
def test_failed_calls_give_back_idle_blocks(program, scenario, where):
    """Every allocation and every queued call of the scenario fails in turn:
    no block goes back to the pool while queued work may use it, and none is
    lost."""
    out = run(program, scenario + where)
    assert out[-1].startswith("done")
    assert not out[:-1], out[:20]


@pytest.mark.parametrize("scenario,edges", [("build_one", 300), ("build", 60000), ("build_bucket", 60000),
                                            ("compute_loop", 60000)])
def test_kept_weights_need_no_room(program, scenario, edges):
    """A build and the loop over the CSR take no more memory than where the
    weights kept for msf_compute are refused theirs."""
    with_weights, without = map(int, run(program, scenario, str(4 * edges))[-1].split())
    assert with_weights == without
