"""The work that a user of the library has it do, as measurable cases.

A case is a dict of plain values; ``prepare`` turns it and a seed into the
inputs on the GPU (and the handle a program would keep), ``run`` makes one
pass through the public entry points and returns all of its outputs.

Calls
  one       ``api.compute``: the forest of one edge list (mask, labels, total)
  batch     ``api.compute_batched``: the forests of many graphs in one call
  train     ``api.msf_weight`` forward and backward: totals, mask, gradients
  session   a ``Graph`` handle built, solved, labelled by connectivity, freed
  min_edge  ``Graph.min_edge`` on a kept handle: one multilinear application

Graphs
  er        uniform random endpoints (self-loops and duplicates kept)
  rmat      R-MAT a,b,c,d = .57,.19,.19,.05; ``permuted``: ids shuffled
  grid      3-D 7-point lattice listed vertex by vertex (road networks)
  mixed     a batch: sizes log-uniform, half uniform random graphs with four
            edges per vertex, half random geometric graphs of mean degree 8

Weights
  unit      float32 odd multiples of 2^-24 in (0, 1)
  normal    float32 standard normal (scores of both signs)
  u32       integers 1..1000 (heavy ties), passed as int32
"""
import math

import numpy as np
import torch

from paper_2110_04865_gb300 import api

DEV = "cuda"


def listed():
    return [
        # a molecule or a cluster of points inside somebody's loop: latency
        {"name": "one_tiny", "call": "one", "graph": "er", "n": 100, "m": 300, "weights": "u32"},
        # the smallest configured workload: a small uniform random graph
        {"name": "one_er4096", "call": "one", "graph": "er", "n": 4096, "m": 32768, "weights": "unit"},
        # a social graph of some 10^4 users with signed scores
        {"name": "one_rmat16", "call": "one", "graph": "rmat", "scale": 16, "m": 1 << 20, "permuted": True,
         "weights": "normal"},
        # the ordinary benchmark graph
        {"name": "one_rmat20", "call": "one", "graph": "rmat", "scale": 20, "m": 16 << 20, "permuted": False,
         "weights": "unit"},
        # no hubs, ragged sizes, integer weights with many ties
        {"name": "one_uniform_odd", "call": "one", "graph": "er", "n": 1000003, "m": 16000057, "weights": "u32"},
        # high diameter and few edges per vertex, as road networks have
        {"name": "one_grid256", "call": "one", "graph": "grid", "nx": 256, "ny": 256, "nz": 256, "weights": "u32"},
        # the largest configured graph on one GPU: 2^30 edges
        {"name": "one_rmat26", "call": "one", "graph": "rmat", "scale": 26, "m": 16 << 26, "permuted": False,
         "weights": "unit"},
        # a small batch of small graphs
        {"name": "batch_64", "call": "batch", "graph": "mixed", "G": 64, "nmin": 64, "nmax": 4096,
         "weights": "unit"},
        # the configured batch: 4096 graphs of 64 to 65536 vertices
        {"name": "batch_4096", "call": "batch", "graph": "mixed", "G": 4096, "nmin": 64, "nmax": 65536,
         "weights": "unit"},
        # a training step that differentiates the forest weights of a batch
        {"name": "train_256", "call": "train", "graph": "mixed", "G": 256, "nmin": 64, "nmax": 8192,
         "weights": "normal"},
        # a program that keeps the graph: build, forest, connectivity, free
        {"name": "session_rmat20", "call": "session", "graph": "rmat", "scale": 20, "m": 16 << 20,
         "permuted": True, "weights": "unit", "csr": False},
        # the kernel that several processes call on their copy of one graph
        {"name": "min_edge_rmat20", "call": "min_edge", "graph": "rmat", "scale": 20, "m": 16 << 20,
         "permuted": False, "weights": "unit"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, nmax):
    kind = rng.choice(["er", "er", "rmat", "rmat", "grid"])
    w = rng.choice(["unit", "normal", "u32"])
    if kind == "er":
        n = _log(rng, 64, nmax)
        return {"graph": "er", "n": n, "m": max(1, int(n * math.exp(rng.uniform(0.0, math.log(32.0))))), "weights": w}
    if kind == "rmat":
        scale = rng.randint(8, max(8, int(math.log2(nmax))))
        m = int((1 << scale) * math.exp(rng.uniform(math.log(2.0), math.log(32.0))))
        return {"graph": "rmat", "scale": scale, "m": m, "permuted": rng.random() < 0.5, "weights": w}
    side = max(4, int(round(nmax ** (1.0 / 3.0))))
    return {"graph": "grid", "nx": _log(rng, 4, side), "ny": _log(rng, 4, side), "nz": _log(rng, 4, side),
            "weights": w}


def draw(rng):
    call = rng.choice(["one", "one", "one", "one", "batch", "batch", "train", "session", "min_edge"])
    if call in ("batch", "train"):
        return {"call": call, "graph": "mixed", "G": _log(rng, 4, 1500), "nmin": _log(rng, 16, 256),
                "nmax": _log(rng, 512, 65536), "weights": rng.choice(["unit", "normal"] if call == "train" else
                                                                    ["unit", "normal", "u32"])}
    c = {"call": call, **_draw_graph(rng, 1 << 22 if call == "one" else 1 << 20)}
    if call == "session":
        c["csr"] = rng.random() < 0.4
    return c


# ---- inputs -------------------------------------------------------------------


def _weights(gen, m, kind):
    if kind == "unit":
        k = torch.randint(0, 1 << 23, (m,), generator=gen, device=DEV, dtype=torch.int32)
        return (k.float() + 0.5) * 2.0 ** -23
    if kind == "normal":
        return torch.randn(m, generator=gen, device=DEV)
    return torch.randint(1, 1001, (m,), generator=gen, device=DEV, dtype=torch.int32)


def _rmat(gen, scale, m, permuted):
    src = torch.empty(m, dtype=torch.int32, device=DEV)
    dst = torch.empty(m, dtype=torch.int32, device=DEV)
    chunk = 1 << 25
    for lo in range(0, m, chunk):
        k = min(chunk, m - lo)
        u = torch.zeros(k, dtype=torch.int32, device=DEV)
        v = torch.zeros(k, dtype=torch.int32, device=DEV)
        for _ in range(scale):
            x = torch.rand(k, generator=gen, device=DEV)
            bu = x >= 0.76
            bv = ((x >= 0.57) ^ bu) | (x >= 0.95)
            u.mul_(2).add_(bu)
            v.mul_(2).add_(bv)
        src[lo:lo + k] = u
        dst[lo:lo + k] = v
    if permuted:
        perm = torch.randperm(1 << scale, generator=gen, device=DEV).to(torch.int32)
        src, dst = perm[src], perm[dst]
    return src, dst


def _grid(nx, ny, nz):
    v = torch.arange(nx * ny * nz, dtype=torch.int32, device=DEV)
    x, y, z = v % nx, (v // nx) % ny, v // (nx * ny)
    ok = torch.stack([x + 1 < nx, y + 1 < ny, z + 1 < nz], 1).reshape(-1)
    step = torch.tensor([1, nx, nx * ny], dtype=torch.int32, device=DEV)
    src = v.repeat_interleave(3)[ok]
    dst = (v[:, None] + step[None, :]).reshape(-1)[ok]
    return src.contiguous(), dst.contiguous()


def _single(case, gen):
    """(n, src, dst) of a one-graph case."""
    if case["graph"] == "er":
        n, m = case["n"], case["m"]
        return n, *(torch.randint(0, n, (m,), generator=gen, device=DEV, dtype=torch.int32) for _ in range(2))
    if case["graph"] == "rmat":
        return 1 << case["scale"], *_rmat(gen, case["scale"], case["m"], case["permuted"])
    return case["nx"] * case["ny"] * case["nz"], *_grid(case["nx"], case["ny"], case["nz"])


def _batch_sizes(case):
    """Vertices of each graph: the quantiles of the log-uniform distribution,
    in order.  Odd ones are geometric graphs, even ones uniform random."""
    q = (np.arange(case["G"]) + 0.5) / case["G"]
    return np.floor(case["nmin"] * (case["nmax"] / case["nmin"]) ** q).astype(np.int64)


def _geometric(gen, sizes):
    """Random geometric graphs in the unit square, r = sqrt(8 / (pi n)), edges
    (i < j) listed by i, then j.  The points are the same for every seed (so
    that the number of edges is); their numbering is not.  Returns (edges per
    graph, src, dst, graph of each edge), local ids, graph by graph."""
    points = torch.Generator(device=DEV)
    points.manual_seed(20211014)
    n = torch.from_numpy(sizes).to(DEV)
    g = torch.repeat_interleave(torch.arange(len(sizes), device=DEV), n)
    base = torch.cumsum(n, 0) - n
    total = int(sizes.sum())
    x, y = torch.rand(2, total, generator=points, device=DEV)
    r = torch.sqrt(8.0 / (math.pi * n.double()))
    r2 = (r * r).float()[g]
    side = torch.clamp(torch.floor(1.0 / r).long(), min=1)
    cells = int((side * side).sum())
    cbase = (torch.cumsum(side * side, 0) - side * side)[g]
    side = side[g]
    cx = torch.minimum((x * side).long(), side - 1)
    cy = torch.minimum((y * side).long(), side - 1)
    cell = cbase + cy * side + cx
    order = torch.argsort(cell, stable=True)
    count = torch.bincount(cell, minlength=cells)  # the last cells may be empty
    start = torch.cumsum(count, 0) - count
    pairs = []
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            i = torch.nonzero((cx + dx >= 0) & (cx + dx < side) & (cy + dy >= 0) & (cy + dy < side))[:, 0]
            c = cell[i] + dy * side[i] + dx
            k, left = 0, count[c]
            first = start[c]
            while True:
                keep = left > k
                if not bool(keep.any()):
                    break
                i, left, first = i[keep], left[keep], first[keep]
                j = order[first + k]
                near = (i < j) & ((x[i] - x[j]) ** 2 + (y[i] - y[j]) ** 2 < r2[i])
                pairs.append((i[near] << 32) | j[near])
                k += 1
    pairs = torch.cat(pairs)
    number = torch.empty(total, dtype=torch.int64, device=DEV)
    shuffled = torch.argsort(g.double() + torch.rand(total, generator=gen, device=DEV, dtype=torch.float64) * 0.999)
    number[shuffled] = torch.arange(total, device=DEV)
    i, j = number[pairs >> 32], number[pairs & 0xFFFFFFFF]
    pairs = torch.sort((torch.minimum(i, j) << 32) | torch.maximum(i, j))[0]
    i, j = pairs >> 32, pairs & 0xFFFFFFFF
    ge = g[i]
    return torch.bincount(ge, minlength=len(sizes)), (i - base[ge]).int(), (j - base[ge]).int(), ge


def _mixed(case, seed, gen):
    """(voff, eoff, src, dst) of a batch, local ids; offsets on the host."""
    sizes = _batch_sizes(case)
    G = len(sizes)
    place = np.random.RandomState(seed % (1 << 32)).permutation(G)  # where each graph stands in the batch
    er, geo = sizes[0::2], sizes[1::2]
    er_at, geo_at = (torch.from_numpy(place[k::2].copy()).to(DEV) for k in (0, 1))
    cnt, gsrc, gdst, gof = _geometric(gen, geo)
    ne = torch.from_numpy(4 * er).to(DEV)
    edges = torch.zeros(G, dtype=torch.int64, device=DEV)
    edges[er_at], edges[geo_at] = ne, cnt
    eoff = torch.zeros(G + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(edges, 0, out=eoff[1:])
    m = int(eoff[-1])
    src = torch.empty(m, dtype=torch.int32, device=DEV)
    dst = torch.empty(m, dtype=torch.int32, device=DEV)
    # the uniform random graphs
    of = torch.repeat_interleave(torch.arange(len(er), device=DEV), ne)
    at = (eoff[er_at] - (torch.cumsum(ne, 0) - ne))[of] + torch.arange(len(of), device=DEV)
    nv = torch.from_numpy(er.copy()).to(DEV)[of]
    for out in (src, dst):
        out[at] = ((torch.randint(0, 1 << 31, (len(of),), generator=gen, device=DEV) * nv) >> 31).int()
    # the geometric ones
    at = (eoff[geo_at] - (torch.cumsum(cnt, 0) - cnt))[gof] + torch.arange(len(gof), device=DEV)
    src[at], dst[at] = gsrc, gdst
    voff = np.zeros(G + 1, np.int64)
    voff[1 + place] = sizes
    return np.cumsum(voff), eoff.cpu().numpy(), src, dst


def _inputs(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    if case["graph"] == "mixed":
        voff, eoff, src, dst = _mixed(case, int(seed), gen)
        s = {"voff": voff, "eoff": eoff, "src": src, "dst": dst}
    else:
        n, src, dst = _single(case, gen)
        s = {"n": n, "src": src, "dst": dst}
    s["w"] = _weights(gen, int(src.shape[0]), case["weights"])
    if case.get("csr"):
        # the symmetric CSR a sparse-matrix program has: both directions of
        # every edge, rows in order (a draw on the diagonal moves off it)
        dst = torch.where(src == dst, (dst + 1) % n, dst)
        rows = torch.cat([src, dst]).long()
        cols = torch.cat([dst, src])
        order = torch.argsort(rows * n + cols, stable=True)
        s["row_ptr"] = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
        torch.cumsum(torch.bincount(rows, minlength=n), 0, out=s["row_ptr"][1:])
        s["src"], s["dst"] = rows[order].int(), cols[order].contiguous()
        s["w"] = torch.cat([s["w"]] * 2)[order].contiguous()
    if case["call"] == "min_edge":
        # trees some rounds on: a seventh of the vertices are roots
        k = max(1, n // 7)
        p = torch.randint(0, k, (n,), generator=gen, device=DEV, dtype=torch.int32)
        p[:k] = torch.arange(k, dtype=torch.int32, device=DEV)
        s["parent"] = p
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["call"] = case["call"]
    if case["call"] == "train":
        G = len(s["voff"]) - 1
        s["w"].requires_grad_(True)
        s["batch"] = api.Batch(s["voff"], s["eoff"], s["src"], s["dst"])
        s["up"] = torch.linspace(0.5, 1.5, G, dtype=torch.float64, device=DEV)
    elif case["call"] == "min_edge":
        s["graph"] = api.Graph(s["n"], s["src"], s["dst"], s["w"])
        del s["src"], s["dst"], s["w"]
    torch.cuda.empty_cache()  # what making the inputs took goes back
    return s


def run(s):
    call = s["call"]
    if call == "one":
        return list(api.compute(s["n"], s["src"], s["dst"], s["w"]))
    if call == "batch":
        return list(api.compute_batched(s["voff"], s["eoff"], s["src"], s["dst"], s["w"]))
    if call == "train":
        totals, mask = api.msf_weight(s["w"], s["batch"])
        (grad,) = torch.autograd.grad(totals, s["w"], s["up"])
        return [totals.detach(), mask, grad]
    if call == "session":
        g = api.Graph(s["n"], s["src"], s["dst"], s["w"], s.get("row_ptr"))
        try:
            return [*g.compute(), g.components()]
        finally:
            g.free()
    return [s["graph"].min_edge(s["parent"])]


def _sizes(case):
    """(vertices, edges, graphs); a geometric graph has about 4 n edges."""
    if case["graph"] == "mixed":
        n = int(_batch_sizes(case).sum())
        return n, 4 * n, case["G"]
    if case["graph"] == "grid":
        x, y, z = case["nx"], case["ny"], case["nz"]
        return x * y * z, (x - 1) * y * z + x * (y - 1) * z + x * y * (z - 1), 1
    return (case["n"] if case["graph"] == "er" else 1 << case["scale"]), case["m"], 1


def work(case):
    n, m, G = _sizes(case)
    if case["call"] in ("one", "batch"):
        b = 12 * m + m + 4 * n + 8 * G  # endpoints and weights; mask, labels, totals
    elif case["call"] == "train":
        b = 12 * m + m + 8 * G + 8 * G + 4 * m  # ...; the incoming and the outgoing gradients
    elif case["call"] == "session":
        slots = 2 * m if case.get("csr") else m
        b = (8 if case.get("csr") else 12) * slots + (8 * n if case.get("csr") else 0) + slots + 4 * n + 8 + 4 * n
    else:
        b = 2 * m * 12 + 4 * n + 8 * n  # both directions of every edge (column and key), parents, minima
    return {"bytes": float(b), "flops": 0.0}


# ---- 64-bit values --------------------------------------------------------------


def _forest(n, src, dst, w):
    """Forest mask by Boruvka's method on 64-bit keys (weight order, index)."""
    m = int(src.shape[0])
    if w.dtype == torch.float32:
        b = (w + 0.0).view(torch.int32).long()
        order = torch.where(b < 0, -(b & 0x7FFFFFFF), b)
    else:
        order = w.long()
    key = (order << 32) + torch.arange(m, device=DEV)
    none = torch.iinfo(torch.int64).max
    label = torch.arange(n, device=DEV)
    ids = torch.arange(n, device=DEV)
    mask = torch.zeros(m, dtype=torch.bool, device=DEV)
    s, d = src.long(), dst.long()
    while True:
        live = s != d
        s, d, key = s[live], d[live], key[live]
        if not len(s):
            return mask
        best = torch.full((n,), none, dtype=torch.int64, device=DEV)
        best.scatter_reduce_(0, s, key, "amin")
        best.scatter_reduce_(0, d, key, "amin")
        root = torch.nonzero(best < none)[:, 0]
        e = best[root] & 0xFFFFFFFF
        mask[e] = True
        a, b = label[src[e].long()], label[dst[e].long()]
        up = ids.clone()
        up[root] = torch.where(a == root, b, a)
        up = torch.where((up[up] == ids) & (ids < up), ids, up)
        while True:
            nxt = up[up]
            if torch.equal(nxt, up):
                break
            up = nxt
        label = up[label]
        s, d = up[s], up[d]


def exact(case, seed):
    n, m, G = _sizes(case)
    if case["call"] == "min_edge" or m > 1 << 28:
        return None
    s = _inputs(case, seed)
    if case["graph"] == "mixed":
        e = torch.from_numpy(np.diff(s["eoff"])).to(DEV)
        g = torch.repeat_interleave(torch.arange(G, device=DEV), e)
        off = torch.from_numpy(s["voff"]).to(DEV)[g]
        src, dst = s["src"] + off, s["dst"] + off
    else:
        g, src, dst = torch.zeros_like(s["src"], dtype=torch.int64), s["src"], s["dst"]
        if case.get("csr"):
            dst = torch.where(src < dst, dst, src)  # a slot below the diagonal is no edge
    mask = _forest(n, src, dst, s["w"])
    totals = torch.zeros(G, dtype=torch.float64, device=DEV)
    totals.index_add_(0, g[mask], s["w"][mask].double())
    if case["call"] == "train":
        up = torch.linspace(0.5, 1.5, G, dtype=torch.float64, device=DEV)
        return [totals, None, up[g] * mask]
    return [None, None, totals, None][:4 if case["call"] == "session" else 3]
