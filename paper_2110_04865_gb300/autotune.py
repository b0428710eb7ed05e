"""Autotuner for the min-edge sweep's tile shape and the compaction threshold.

With the library's default options msf_compute and msf_compute_batched run no
sweep (they solve from the edges), and an option that asks for another sweep
form or threshold would put the round loop in their place.  What is tuned then
is msf_min_edge: for a built graph one sweep (p = identity, every slot live) is
timed for every tile shape of its own form -- slots per lane (tile width
32*V), resident blocks per SM -- and the fastest is set as the library's
process-wide option, the library's default on a near-tie.  The batched form
has nothing to tune.

Where the other options select the round loop (a schedule, a builder, a kernel
form, the host-driven loop, a lower limit), the whole loop is timed
(msf_compute, msf_compute_batched), or one sweep, for every combination of
sweep form (register tiles, with or without next-tile prefetch; the
shared-memory pipeline; the register pipeline), slots per lane and resident
blocks per SM, then the compaction thresholds in TAU_CANDIDATES with the
fastest shape (compaction pays only when enough rounds follow on a much
smaller edge list).

A sweep's duration comes from the library itself (CUDA events around that
launch only, ``msf_stats.min_edge_ms``).  Results are cached per device, graph
class (log2 of the slot count, rounded average degree) and what was tuned in
``_build/autotune.json`` next to the library; entries of another FORMAT are
not read.
"""
from __future__ import annotations

import json
import math
import os
import statistics

import torch

from . import _abi

CACHE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "_build", "autotune.json")
# (slots per lane, prefetch, blocks per SM, sweep form)
CANDIDATES = ([(spl, pf, bps, 0) for spl in (4, 8, 16) for pf in (0, 1) for bps in (2, 4, 8)]
              + [(spl, 0, bps, 1) for spl in (4, 8, 16) for bps in (1, 2, 3, 4)]
              + [(spl, 0, bps, 2) for spl in (4, 8) for bps in (2, 3, 4)])
SHAPE_KEYS = ("spl", "prefetch", "blocks_per_sm", "sweep")
CONFIG_KEYS = SHAPE_KEYS + ("compact_tau",)
# compaction thresholds, the library's default first (kept on near-ties)
TAU_CANDIDATES = (0.5, 0.25, 0.0)
# shapes of msf_min_edge's own sweep, the library's default first; it knows no
# prefetch, and from four slots a row on takes 8 a lane for 4
MIN_EDGE_CANDIDATES = [(4, 0, 4, 0)] + [(spl, 0, bps, 0) for spl in (4, 8, 16) for bps in (2, 4, 8)
                                        if (spl, bps) != (4, 4)]
FORMAT = 2  # of the cache's entries: 1 chose by calls that the options no longer reach


def pick_shape(table):
    """The shape to keep from rows (ms, sweep_ms, spl, prefetch, blocks_per_sm,
    sweep): the fastest by ms; among the rows within 1 % of it (closer than
    the measurements' noise), the one whose full sweep is fastest."""
    fastest = min(t[0] for t in table)
    return min((t for t in table if t[0] <= 1.01 * fastest), key=lambda t: t[1])


def pick_first(rows):
    """The first row, in candidate order, whose time (its first field) is
    within 1 % of the fastest: an earlier candidate wins a near-tie (for the
    compaction thresholds the library's default comes first)."""
    fastest = min(r[0] for r in rows)
    return next(r for r in rows if r[0] <= 1.01 * fastest)


def _key(device: torch.device, st) -> str:
    name = torch.cuda.get_device_name(device).replace(" ", "_")
    cls = int(round(math.log2(max(int(st.nnz), 1))))
    deg = int(round(st.nnz / max(int(st.rows), 1)))
    deg_cls = int(round(math.log2(max(deg, 1))))
    return f"{name}/nnz2^{cls}/deg2^{deg_cls}"


def _load_cache() -> dict:
    try:
        return json.load(open(CACHE))
    except (OSError, ValueError):
        return {}


def apply(cfg: dict):
    _abi.msf_set_option(_abi.OPT_SLOTS_PER_LANE, cfg["spl"])
    _abi.msf_set_option(_abi.OPT_PREFETCH, cfg["prefetch"])
    _abi.msf_set_option(_abi.OPT_BLOCKS_PER_SM, cfg["blocks_per_sm"])
    _abi.msf_set_option(_abi.OPT_SWEEP, cfg.get("sweep", 0))
    if "compact_tau" in cfg:
        _abi.msf_set_option(_abi.OPT_COMPACT_TAU, cfg["compact_tau"])


def round_loop_selected() -> bool:
    """Whether the options that are not tuned here put the round loop in the
    place of the solvers from the edges."""
    g = _abi.msf_get_option
    return (any(g(o) != 0 for o in (_abi.OPT_EXEC_MODE, _abi.OPT_SHORTCUT, _abi.OPT_KERNEL, _abi.OPT_BUILD))
            or g(_abi.OPT_ROUND_LIMIT) < 64 or g(_abi.OPT_JUMP_LIMIT) < 64)


def _save(cache: dict):
    try:
        os.makedirs(os.path.dirname(CACHE), exist_ok=True)
        tmp = CACHE + f".tmp{os.getpid()}"
        json.dump(cache, open(tmp, "w"), indent=1)
        os.replace(tmp, CACHE)
    except OSError:
        pass


class _Timer:
    """Times calls on the current stream, the L2 flushed before each."""

    def __init__(self, dev, flush_bytes: int):
        self.flush = torch.empty(flush_bytes, dtype=torch.uint8, device=dev)
        self.stream = torch.cuda.current_stream(dev)

    def call_ms(self, call, reps: int) -> float:
        call()  # warm-up (and graph instantiation for a new shape)
        ts = []
        for _ in range(reps):
            self.flush.fill_(1)
            a = torch.cuda.Event(enable_timing=True)
            b = torch.cuda.Event(enable_timing=True)
            a.record(self.stream)
            call()
            b.record(self.stream)
            b.synchronize()
            ts.append(a.elapsed_time(b))
        return statistics.median(ts)

    def sweep_ms(self, graph, parent, reps: int) -> float:
        graph.min_edge(parent)  # warm-up
        ts = []
        for _ in range(reps):
            self.flush.fill_(1)
            graph.min_edge(parent)
            ts.append(float(graph.stats().min_edge_ms))
        return statistics.median(ts)


def tune(graph, reps: int = 5, use_cache: bool = True, flush_bytes: int = 256 << 20,
         objective: str = "compute") -> dict:
    """Times the candidates on `graph` (an api.Graph) and applies the fastest.
    With the round loop selected, objective "compute" is the whole loop
    (msf_compute, edge mask only; later rounds, where parents repeat, weigh in)
    and "sweep" one min-edge sweep with every slot live; otherwise msf_compute
    does not depend on the shape and the sweep decides (``ms`` is then
    msf_compute's time for "compute").  Returns dict(spl, prefetch,
    blocks_per_sm, sweep, compact_tau, ms, sweep_ms, table)."""
    dev = graph.device if graph.device is not None else torch.device("cuda", torch.cuda.current_device())
    loop = round_loop_selected()
    key = _key(dev, graph.stats()) + f"/{objective}/{'loop' if loop else 'edges'}/{FORMAT}"
    cache = _load_cache()
    if use_cache and key in cache:
        apply(cache[key])
        return dict(cache[key], cached=True)
    parent = torch.arange(graph.n, dtype=torch.int32, device=dev)
    timer = _Timer(dev, flush_bytes)
    compute = lambda: graph.compute(mask=True, labels=False, total=False)  # noqa: E731
    table = []
    for spl, pf, bps, sw in CANDIDATES if loop else MIN_EDGE_CANDIDATES:
        apply(dict(spl=spl, prefetch=pf, blocks_per_sm=bps, sweep=sw))
        ms = timer.call_ms(compute, max(reps, 3)) if loop and objective == "compute" else None
        sweep_ms = timer.sweep_ms(graph, parent, reps)
        table.append((sweep_ms if ms is None else ms, sweep_ms, spl, pf, bps, sw))
    ms, sweep_ms, spl, pf, bps, sw = pick_shape(table) if loop else pick_first(table)
    best = dict(spl=spl, prefetch=pf, blocks_per_sm=bps, sweep=sw, ms=ms, sweep_ms=sweep_ms)
    if not loop:
        best.update(compact_tau=TAU_CANDIDATES[0])
        if objective == "compute":
            apply(best)
            best.update(ms=timer.call_ms(compute, max(reps, 3)))
    elif objective == "compute":
        # the compaction threshold with that shape; an earlier candidate wins
        # a near-tie
        ttimes = []
        for tau in TAU_CANDIDATES:
            apply(dict(best, compact_tau=tau))
            ttimes.append((timer.call_ms(compute, max(reps, 3)), tau))
        t_ms, tau = pick_first(ttimes)
        best.update(compact_tau=tau, ms=t_ms)
    else:
        best.update(compact_tau=_abi.msf_get_option(_abi.OPT_COMPACT_TAU))
    apply(best)
    cache[key] = best
    _save(cache)
    return dict(best, cached=False,
                table=[dict(ms=t, sweep_ms=u, spl=a, prefetch=b, blocks_per_sm=c, sweep=e)
                       for t, u, a, b, c, e in table])


def tune_batched(call, key: str, reps: int = 3, use_cache: bool = True, flush_bytes: int = 256 << 20,
                 device=None) -> dict:
    """The same for the batched form: `call()` enqueues one msf_compute_batched
    call on the current stream (the whole batch: build and round loop).  With
    the round loop selected every sweep shape is timed on it, then the
    compaction thresholds with the fastest shape; otherwise the call depends on
    none of them and is timed as the options stand (a sweep form or threshold
    off its default goes back to it).  `key` names the batch class for the
    cache.  Returns dict(spl, prefetch, blocks_per_sm, sweep, compact_tau, ms)."""
    dev = device if device is not None else torch.device("cuda", torch.cuda.current_device())
    loop = round_loop_selected()
    name = torch.cuda.get_device_name(dev).replace(" ", "_")
    ckey = f"{name}/batched/{key}/{'loop' if loop else 'edges'}/{FORMAT}"
    cache = _load_cache()
    if use_cache and ckey in cache:
        apply(cache[ckey])
        return dict(cache[ckey], cached=True)
    timer = _Timer(dev, flush_bytes)
    if loop:
        tau0 = _abi.msf_get_option(_abi.OPT_COMPACT_TAU)
        table = []
        for spl, pf, bps, sw in CANDIDATES:
            apply(dict(spl=spl, prefetch=pf, blocks_per_sm=bps, sweep=sw, compact_tau=tau0))
            table.append((timer.call_ms(call, reps), spl, pf, bps, sw))
        ms, spl, pf, bps, sw = pick_first(table)
        best = dict(spl=spl, prefetch=pf, blocks_per_sm=bps, sweep=sw)
        ttimes = []
        for tau in TAU_CANDIDATES:
            apply(dict(best, compact_tau=tau))
            ttimes.append((timer.call_ms(call, reps), tau))
        t_ms, tau = pick_first(ttimes)
        best.update(compact_tau=tau, ms=t_ms)
    else:
        best = dict(spl=int(_abi.msf_get_option(_abi.OPT_SLOTS_PER_LANE)),
                    prefetch=int(_abi.msf_get_option(_abi.OPT_PREFETCH)),
                    blocks_per_sm=int(_abi.msf_get_option(_abi.OPT_BLOCKS_PER_SM)), sweep=0,
                    compact_tau=TAU_CANDIDATES[0])
        apply(best)
        best.update(ms=timer.call_ms(call, reps))
    apply(best)
    cache[ckey] = best
    _save(cache)
    return dict(best, cached=False)
