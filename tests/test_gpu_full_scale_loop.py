"""The round loop over the CSR and one min-edge sweep at full size: R-MAT scale 26
(2^26 vertices, 2^30 edges, about 2.15e9 slots, built through sub-buckets), which
the default calls solve from the edges.  The loop's forest is the solvers' (which
the full oracle covers at this size), in two launch shapes; the sweep's minima
are those of the edge list.  Needs about 90 GB of device memory."""
from __future__ import annotations

import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.slow]

SCALE, M = 26, 1 << 30


def rmat(torch, gen):
    """R-MAT endpoints (a, b, c, d = .57, .19, .19, .05), drawn on the GPU."""
    src, dst = (torch.empty(M, dtype=torch.int32, device="cuda") for _ in range(2))
    step = 1 << 25
    for lo in range(0, M, step):
        u, v = (torch.zeros(step, dtype=torch.int32, device="cuda") for _ in range(2))
        for _ in range(SCALE):
            x = torch.rand(step, generator=gen, device="cuda")
            bu = x >= 0.76
            bv = ((x >= 0.57) ^ bu) | (x >= 0.95)
            u.mul_(2).add_(bu)
            v.mul_(2).add_(bv)
        src[lo:lo + step], dst[lo:lo + step] = u, v
    return src, dst


def test_rmat26_loop_and_sweep():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_04865_gb300 import _abi, api, autotune, build_lib
    build_lib.build()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(26)
    n = 1 << SCALE
    src, dst = rmat(torch, gen)
    w = (torch.randint(0, 1 << 23, (M,), generator=gen, device="cuda", dtype=torch.int32).float() + 0.5) * 2.0 ** -23
    old = {o: _abi.msf_get_option(o) for o in range(15)}
    g = api.Graph(n, src, dst, w)
    try:
        want, solved = g.compute(), g.stats()
        for shape in (dict(spl=4, prefetch=0, blocks_per_sm=4), dict(spl=4, prefetch=1, blocks_per_sm=8)):
            autotune.apply(dict(shape, sweep=0, compact_tau=0.25))  # a threshold of its own selects the loop
            got, st = g.compute(), g.stats()
            assert st.rounds == solved.rounds and st.kernels > solved.kernels + 8 * st.rounds, shape
            for a, b in zip(got, want):
                assert torch.equal(a, b), shape
            del got
        assert g.stats().nnz > 1 << 30  # (slots beyond 32-bit counts of bytes, near 2^31 of them)
        # the sweep: the smallest (weight, edge) at each vertex; weights are positive
        # floats, ordered by their bits, and their order words have the top bit set
        r = g.min_edge(torch.arange(n, dtype=torch.int32, device="cuda"))
    finally:
        for o, v in old.items():
            _abi.msf_set_option(o, v)
        g.free()
    del want
    torch.cuda.empty_cache()
    none = torch.iinfo(torch.int64).max
    least = torch.full((n,), none, dtype=torch.int64, device="cuda")
    step = 1 << 27
    for lo in range(0, M, step):
        s, d = src[lo:lo + step].long(), dst[lo:lo + step].long()
        key = (w[lo:lo + step].view(torch.int32).long() << 32) | torch.arange(lo, lo + step, device="cuda")
        key = torch.where(s == d, none, key)
        least.scatter_reduce_(0, s, key, "amin")
        least.scatter_reduce_(0, d, key, "amin")
        del s, d, key
    assert torch.equal(r & none, least) and bool((r < 0).all())
