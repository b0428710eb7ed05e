// Forests of small graphs, one thread block per graph.
//
// A graph whose parents (16 bits a vertex), component minima (64 bits a
// vertex) and forest bitmap (a bit an edge) fit in one SM's shared memory is
// solved by one block in one launch: a call on a small graph is one launch
// instead of some sixty, and the graphs of a batch run side by side, one block
// each, largest first.  The method is the one of solve.cu -- light edges first
// by a sampled threshold, Boruvka rounds on them, a filter pass over the edges,
// rounds on the edges left -- with block barriers for the grid barriers and
// shared memory for every gather (a random 32-lane gather costs 3 to 4 bank
// conflicts there, 32 wavefronts in L1).  Graphs of at most KEEP edges a thread
// stay in registers from the first read to the result; larger ones keep lists
// in global scratch (mostly L2), which move to registers once they are short.
//
// What bounds it is latency: a round is four block barriers with a chain of
// shared-memory accesses between them (about 5 us at 4096 vertices and 1024
// threads, half of it the settling pass and the marks), a pass over 32 768
// edges is 8 batches per warp (7 us).  Variants that measured slower: 64-bit
// minima by compare-and-swap (ER 4096 112 us against 85), 512 threads with 128
// registers (125), chains followed inside the minimum pass (115).
//
// Whole calls (CSR path before, this after): 100 vertices 293 -> 35 us, ER 4096
// 391 -> 97, a batch of 64 graphs 590 -> 90, forward and backward of 256 graphs
// 1120 -> 351 (the rest of it is the autograd engine).
#include <cstring>
#include <mutex>

#include "exact.cuh"
#include "internal.cuh"

namespace msf {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int ROUND_CAP = 64;  // Boruvka rounds at most (components at least halve)
constexpr int HOPS = 16;       // hops of one settling pass

struct SmallArgs {
  const int32_t *src, *dst;
  const int2 *ends;        // instead of src and dst: validated ends
  const uint32_t *w;
  int32_t wtype;
  int32_t count;           // the loop's rounds are counted (no edges filtered)
  int32_t vec;             // the three arrays are 16-byte aligned
  const int64_t *voff, *eoff;  // [2 * block]: its graph's offsets (pinned host memory, read in place)
  const int32_t *order;    // graph of each block, or NULL
  const int64_t *loff;     // first list entry of each block's graph, or NULL
  int64_t n, m;            // one graph
  uint4 *list;             // kept edges
  uint8_t *mask;
  int32_t *labels;
  double *totals;
  unsigned *host;          // pinned: [0] index out of range, [1] NaN weight, [2..4] LoopCounts
};

// Dynamic shared memory of a graph: minima, parents, forest bitmap.
__host__ __device__ inline size_t small_smem(int64_t n, int64_t m) {
  const int64_t nn = (n + 3) / 4 * 4;
  return (size_t)nn * 10 + (size_t)((m + 31) / 32 + 2) * 4;
}

// Light edges kept per vertex, for graphs of several times as many edges.
constexpr double LIGHT = 1.5;
// List entries a lane keeps in registers.
constexpr int KEEP = 8;

// Entries: endpoints (roots) u | v << 16, edge, ordered weight.
template <int NT, bool F32>
__global__ void __launch_bounds__(NT, 1024 / NT) k_small(SmallArgs A) {
  constexpr int NW = NT / 32;
  constexpr uint32_t NONE = 0xffffffffu;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ BlockSums sums;
  __shared__ long long sbins[256];
  __shared__ unsigned long long s_usum, s_thresh;
  __shared__ unsigned s_pairs[2], s_edges;  // trees formed, by round modulo 2; forest edges
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned below = (1u << lane) - 1u;
  const int at = 2 * (int)blockIdx.x;
  const int g = A.order ? A.order[blockIdx.x] : 0;
  const int64_t v0 = A.order ? A.voff[at] : 0, e0 = A.order ? A.eoff[at] : 0;
  const int n = (int)(A.order ? A.voff[at + 1] - v0 : A.n);
  const int64_t e1 = A.order ? A.eoff[at + 1] : A.m;
  const int m = (int)(e1 - e0);
  const int nn = (n + 3) / 4 * 4;
  // a component's minimum: its smallest weight, then the smallest edge of that
  // weight (two 32-bit minima, each one native shared atomic; a 64-bit
  // minimum is a compare-and-swap loop)
  uint32_t *rw = reinterpret_cast<uint32_t *>(raw), *re = rw + nn;
  uint16_t *p = reinterpret_cast<uint16_t *>(re + nn);
  uint32_t *bits = reinterpret_cast<uint32_t *>(p + nn);
  for (int v = threadIdx.x; v < n; v += NT) {
    p[v] = (uint16_t)v;
    rw[v] = re[v] = NONE;
  }
  for (int i = threadIdx.x; i < (m + 31) / 32 + 2; i += NT) bits[i] = 0u;
  sums.clear();
  if (threadIdx.x == 0) s_usum = s_edges = 0;
  int hooked = 0;  // rounds with hooks
  unsigned long long usum = 0;  // uint32 weights of the thread's forest edges
  uint32_t top = 0;             // largest endpoint seen
  bool nan = false;
  uint32_t kuv[KEEP], ke[KEEP], kw[KEEP];  // kept entries; kuv = 0: none left

  auto mark = [&](uint32_t e, uint32_t ow) {
    const uint32_t le = e - (uint32_t)e0;
    atomicOr(bits + (le >> 5), 1u << (le & 31u));
    if (F32) sums.add(ow);
    else usum += ow;
  };
  // hook along a minimum (tie breaking as in Algorithm 2: of two roots that
  // chose the same edge the smaller stays a root)
  unsigned pairs = 0;  // roots of the thread's edges that chose each other
  auto hook = [&](uint32_t uv, uint32_t e, uint32_t ow) -> bool {
    const uint32_t u = uv & 0xffffu, v = uv >> 16;
    const bool mu = rw[u] == ow && re[u] == e, mv = rw[v] == ow && re[v] == e;
    if (!(mu || mv)) return false;
    pairs += mu && mv;
    if (mu && (!mv || v < u)) p[u] = (uint16_t)v;
    else p[v] = (uint16_t)u;
    return true;
  };
  auto relabel = [&](uint32_t uv) -> uint32_t {
    const uint32_t u = p[uv & 0xffffu], v = p[uv >> 16];
    return u == v ? 0u : u | (v << 16);
  };
  auto min_weight = [&](uint32_t uv, uint32_t ow) {
    atomicMin(rw + (uv & 0xffffu), ow);
    atomicMin(rw + (uv >> 16), ow);
  };
  auto min_edge = [&](uint32_t uv, uint32_t e, uint32_t ow) {
    const uint32_t u = uv & 0xffffu, v = uv >> 16;
    if (rw[u] == ow) atomicMin(re + u, e);
    if (rw[v] == ow) atomicMin(re + v, e);
  };
  // A round's hooks are counted (its slot was cleared before its first barrier).
  auto count_round = [&]() {
    if (!A.count) return;
    const unsigned t = __reduce_add_sync(FULL, pairs);
    if (lane == 0 && t) atomicAdd(&s_pairs[hooked & 1], t);
    pairs = 0;
    ++hooked;
  };
  // Every parent a root (a vertex's parent is written by its own thread only),
  // the minima cleared; four vertices' chains side by side, in passes of up to
  // HOPS hops: the next pass starts from where the others have got to, so that a
  // chain of k hops takes log k passes (a path with rising weights hooks as one
  // chain, which took a thread half its length: 5.1 ms of a compute on 20 000
  // vertices).  One pass is enough for most rounds, and its barrier is the one
  // that ends the round.
  auto settle = [&]() {
    constexpr int U = 4;
    volatile uint16_t *q = p;
    bool more, first = true;
    do {
      more = false;
      for (int v = threadIdx.x; v < n; v += U * NT) {
        uint32_t x[U], y[U];
#pragma unroll
        for (int j = 0; j < U; ++j) x[j] = v + j * NT < n ? q[v + j * NT] : 0u;
#pragma unroll
        for (int j = 0; j < U; ++j) y[j] = q[x[j]];
        if (first) {
#pragma unroll
          for (int j = 0; j < U; ++j)
            if (v + j * NT < n) rw[v + j * NT] = re[v + j * NT] = NONE;
        }
        bool on = false;
#pragma unroll
        for (int j = 0; j < U; ++j) on |= x[j] != y[j];
        if (!on) continue;
        for (int h = 0; h < HOPS && on; ++h) {
          on = false;
#pragma unroll
          for (int j = 0; j < U; ++j) {
            const uint32_t z = q[y[j]];
            on |= z != y[j];
            y[j] = z;
          }
        }
        more |= on;
#pragma unroll
        for (int j = 0; j < U; ++j)
          if (v + j * NT < n) q[v + j * NT] = (uint16_t)y[j];
      }
      first = false;
    } while (__syncthreads_or(more));
  };
  // Rounds on the entries in registers until none joins two trees.  The forest
  // edges are marked and summed once at the end.
  auto rounds_kept = [&]() {
    unsigned in = 0;  // kept entries in the forest
    for (int k = 0; k < ROUND_CAP; ++k) {
      uint32_t left = 0;
      if (threadIdx.x == 0) s_pairs[hooked & 1] = 0;
#pragma unroll
      for (int j = 0; j < KEEP; ++j) {
        if (!kuv[j]) continue;
        kuv[j] = relabel(kuv[j]);
        if (kuv[j]) min_weight(kuv[j], kw[j]);
        left |= kuv[j];
      }
      if (!__syncthreads_or(left != 0)) break;
#pragma unroll
      for (int j = 0; j < KEEP; ++j)
        if (kuv[j]) min_edge(kuv[j], ke[j], kw[j]);
      __syncthreads();
#pragma unroll
      for (int j = 0; j < KEEP; ++j)
        if (kuv[j] && hook(kuv[j], ke[j], kw[j])) {
          in |= 1u << j;
          kuv[j] = 0u;
        }
      count_round();
      __syncthreads();
      settle();
    }
#pragma unroll
    for (int j = 0; j < KEEP; ++j)
      if (in >> j & 1u) mark(ke[j], kw[j]);
  };
  // The warp's list lies in the places of its batches of 128 edges, batch k of warp
  // w the one w + k * NW of the graph: an input sorted by weight, or with one
  // weight for all, has its light edges side by side, and one run of edges per
  // warp gave nearly all of them to one (2 graphs of 4000 vertices and 400 000
  // sorted edges 850 us, now 257; with weights in any order 2 % more than runs,
  // R-MAT 12 with 105 000 edges 150 -> 157).
  auto place = [&](int i) { return (((i >> 7) * NW + wid) << 7) | (i & 127); };
  // Rounds on the warp's list; one of at most KEEP entries a lane goes to
  // registers first.
  uint4 *L = nullptr;
  auto rounds = [&](int cnt) {
    constexpr int U = 4;
    for (int k = 0; k < ROUND_CAP; ++k) {
      if (__syncthreads_and(cnt <= 32 * KEEP)) {
#pragma unroll
        for (int j = 0; j < KEEP; ++j) {
          const int i = j * 32 + lane;
          const uint4 x = i < cnt ? L[place(i)] : make_uint4(0u, 0u, 0u, 0u);
          kuv[j] = x.x;
          ke[j] = x.z;
          kw[j] = x.w;
        }
        rounds_kept();
        return;
      }
      int out = 0;
      if (threadIdx.x == 0) s_pairs[hooked & 1] = 0;
      for (int b0 = 0; b0 < cnt; b0 += 32 * U) {  // (a batch)
        const uint4 *Lb = L + place(b0);
        uint4 x[U];
#pragma unroll
        for (int j = 0; j < U; ++j) x[j] = b0 + j * 32 + lane < cnt ? Lb[j * 32 + lane] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int j = 0; j < U; ++j) {
          if (x[j].x) x[j].x = relabel(x[j].x);
          const unsigned bal = __ballot_sync(FULL, x[j].x != 0);
          if (x[j].x) {
            min_weight(x[j].x, x[j].w);
            L[place(out + __popc(bal & below))] = x[j];
          }
          out += __popc(bal);
        }
      }
      __syncwarp();
      cnt = out;
      if (!__syncthreads_or(cnt > 0)) return;
      for (int b0 = 0; b0 < cnt; b0 += 32 * U) {  // (a batch)
        const uint4 *Lb = L + place(b0);
        uint4 x[U];
#pragma unroll
        for (int j = 0; j < U; ++j) x[j] = b0 + j * 32 + lane < cnt ? Lb[j * 32 + lane] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int j = 0; j < U; ++j)
          if (x[j].x) min_edge(x[j].x, x[j].z, x[j].w);
      }
      __syncthreads();
      for (int b0 = 0; b0 < cnt; b0 += 32 * U) {  // (a batch)
        const uint4 *Lb = L + place(b0);
        uint4 x[U];
#pragma unroll
        for (int j = 0; j < U; ++j) x[j] = b0 + j * 32 + lane < cnt ? Lb[j * 32 + lane] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int j = 0; j < U; ++j)
          if (x[j].x && hook(x[j].x, x[j].z, x[j].w)) mark(x[j].z, x[j].w);
      }
      count_round();
      __syncthreads();
      settle();
    }
  };
  // An invalid edge ends the call: its index must not be used.
  auto invalid = [&]() -> bool {
    const bool bad = m > 0 && top >= (uint32_t)n;
    if (bad) A.host[0] = 1u;
    if (nan) A.host[1] = 1u;
    return __syncthreads_or(bad || nan);
  };

  if (m <= KEEP * NT) {
    // the whole graph in registers
#pragma unroll
    for (int j = 0; j < KEEP; ++j) {
      const int i = j * NT + threadIdx.x;
      uint32_t u = 0, v = 0, w = 0;
      if (i < m) {
        const int2 uv = A.ends ? A.ends[e0 + i] : make_int2(A.src[e0 + i], A.dst[e0 + i]);
        u = (uint32_t)uv.x;
        v = (uint32_t)uv.y;
        w = A.w[e0 + i];
      }
      top = max(top, max(u, v));
      nan |= F32 && (w << 1) > 0xff000000u;
      kuv[j] = u == v ? 0u : u | (v << 16);
      ke[j] = (uint32_t)(e0 + i);
      kw[j] = ord_weight_dev(w, F32 ? MSF_F32 : MSF_U32);
    }
    if (invalid()) return;
    rounds_kept();
  } else {
    // The threshold: about the key of the wanted rank in a sample of warp 0,
    // found bit by bit with ballots -- as a rule twelve bits below the samples'
    // common prefix; any threshold is a valid one.
    const bool filter = !A.count && (float)m > (float)(1.5 * LIGHT) * (float)n;
    if (wid == 0 && filter) {
      constexpr int PER = 8;
      uint32_t w[PER], e[PER], lo = NONE, up = 0u;
#pragma unroll
      for (int j = 0; j < PER; ++j) {
        const int64_t i = (int64_t)(lane * PER + j) * m / (32 * PER);
        e[j] = (uint32_t)(e0 + i);
        w[j] = ord_weight_dev(A.w[e0 + i], A.wtype);
        lo = min(lo, w[j]);
        up = max(up, w[j]);
      }
      lo = __reduce_min_sync(FULL, lo);
      up = __reduce_max_sync(FULL, up);
      const int rank = light_rank(LIGHT, n, m, 32 * PER, 8);
      auto below_key = [&](uint32_t tw, uint32_t te) {
        int c = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j) c += __popc(__ballot_sync(FULL, w[j] < tw || (w[j] == tw && e[j] < te)));
        return c;
      };
      const int high = 31 - __clz((int)((lo ^ up) | 1u));  // the highest bit in which samples differ
      uint32_t tw = high >= 31 ? 0u : lo >> (high + 1) << (high + 1), te = NONE;
      auto refine = [&](int from, int to) {
        for (int b = from; b >= 0 && b > to; --b) {
          const uint32_t c = tw | (1u << b);
          if (below_key(c, 0u) <= rank) tw = c;
        }
      };
      refine(high, high - 12);
      if (high >= 12) {
        // all weights with these bits, unless many samples share them (a few
        // weights of which the others are exact multiples, negative ones): by the
        // other bits too.  None of them, where -1 and 1 are the only weights, left
        // no edge light (40 graphs of 4000 vertices and 400 000 edges 2.6 ms, now 0.36)
        const uint32_t up = tw | ((2u << (high - 12)) - 1u);
        if (below_key(up, NONE) <= rank + rank / 4 + 1) tw = up;
        else refine(high - 12, -1);
      }
      if (below_key(tw, NONE) > rank + rank / 4 + 1) {  // many ties: by edge index
        te = 0;
        for (int b = 31; b >= 0; --b) {
          const uint32_t c = te | (1u << b);
          if (below_key(tw, c) <= rank) te = c;
        }
        te &= ~127u;  // (batches start at multiples of 128)
      }
      if (lane == 0) s_thresh = ((unsigned long long)tw << 32) | te;
    }
    __syncthreads();
    Limit<F32> limit(filter ? s_thresh : KEY_INF);

    // the warp's batches of 128 edges (indices from the first batch on)
    const int64_t a0 = e0 & ~(int64_t)127;
    const int first = (int)(e0 - a0), end = (int)(e1 - a0);
    const int batches = (end + 127) >> 7, mine = wid < batches ? ((batches - wid + NW - 1) / NW) << 7 : 0;
    const int32_t *S = A.src + a0, *D = A.dst + a0;
    const uint32_t *W = A.w + a0;
    const bool vec = A.vec != 0;
    L = A.list + (A.loff ? A.loff[blockIdx.x] : 0);
    int cnt = 0;
    {
      auto load = [&](int k) {
        const int i = place(k) + 4 * lane, hi = k < mine ? end : 0;
        return A.ends ? pair_quad(A.ends, W, i, hi) : edge_quad<true>(S, D, W, vec, i, first, hi);
      };
      auto body = [&](const EdgeQuad &q, int k) {
        const int b = place(k), i = b + 4 * lane;
        limit.batch(a0 + b);
        const uint32_t u[4] = {(uint32_t)q.s.x, (uint32_t)q.s.y, (uint32_t)q.s.z, (uint32_t)q.s.w};
        const uint32_t v[4] = {(uint32_t)q.d.x, (uint32_t)q.d.y, (uint32_t)q.d.z, (uint32_t)q.d.w};
        const uint32_t w[4] = {q.w.x, q.w.y, q.w.z, q.w.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          top = max(top, max(u[j], v[j]));
          if (F32) nan |= __uint_as_float(w[j]) != __uint_as_float(w[j]);
          const bool sel = limit.below(w[j]) && u[j] != v[j];
          const unsigned bal = __ballot_sync(FULL, sel);
          if (sel)
            L[place(cnt + __popc(bal & below))] = make_uint4(u[j] | (v[j] << 16), 0u, (uint32_t)a0 + (uint32_t)(i + j),
                                                      ord_weight_dev(w[j], F32 ? MSF_F32 : MSF_U32));
          cnt += __popc(bal);
        }
      };
      stream2<EdgeQuad>(0, mine, load, body);
      __syncwarp();
    }
    if (invalid()) return;
    rounds(cnt);
    if (filter) {
      // the edges between components (the heavy ones: a light edge lies inside)
      cnt = 0;
      auto load = [&](int k) {
        return edge_quad<false>(S, D, W, vec, place(k) + 4 * lane, first, k < mine ? end : 0);
      };
      auto body = [&](const EdgeQuad &q, int k) {
        const int i = place(k) + 4 * lane;
        const uint32_t u[4] = {p[q.s.x], p[q.s.y], p[q.s.z], p[q.s.w]};
        const uint32_t v[4] = {p[q.d.x], p[q.d.y], p[q.d.z], p[q.d.w]};
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = u[j] != v[j] ? W[i + j] : 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const bool sel = u[j] != v[j];
          const unsigned bal = __ballot_sync(FULL, sel);
          if (sel)
            L[place(cnt + __popc(bal & below))] = make_uint4(u[j] | (v[j] << 16), 0u, (uint32_t)a0 + (uint32_t)(i + j),
                                                      ord_weight_dev(w[j], F32 ? MSF_F32 : MSF_U32));
          cnt += __popc(bal);
        }
      };
      stream2<EdgeQuad>(0, mine, load, body);
      __syncwarp();
      rounds(cnt);
    }
  }
  if (A.count) {
    __syncthreads();
    unsigned c = 0;
    for (int i = threadIdx.x; i < (m + 31) / 32; i += NT) c += __popc(bits[i]);
    c = __reduce_add_sync(FULL, c);
    if (lane == 0 && c) atomicAdd(&s_edges, c);
    __syncthreads();
    if (threadIdx.x == 0) {
      A.host[2] = (unsigned)hooked;
      A.host[3] = hooked ? s_pairs[(hooked - 1) & 1] : 0u;
      A.host[4] = s_edges;
    }
  }
  // Results (parents are roots, the minima clear).  The last warp rounds the
  // total while the others write labels and mask.
  if (A.totals && !F32) {
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) usum += __shfl_xor_sync(FULL, usum, d);
    if (lane == 0 && usum) atomicAdd(&s_usum, usum);
  }
  __syncthreads();  // every warp's marks and weights are in (rounds_kept makes them last)
  if (wid == NW - 1) {
    if (!A.totals) return;
    if (F32) {
#pragma unroll
      for (int i = 0; i < 8; ++i) sbins[lane + 32 * i] = (long long)sums.get(lane + 32 * i);
      __syncwarp();
      const double t = combine_bins_warp(sbins, MSF_F32);
      if (lane == 0) A.totals[g] = t;
    } else if (lane == 0) {
      A.totals[g] = __ull2double_rn(s_usum);
    }
    return;
  }
  constexpr int NO = NT - 32;  // the other warps
  if (A.labels) {
    // the smallest vertex of every tree, in rw (the root itself is added when
    // read)
    for (int b = wid * 32; b < n; b += NO) {
      const int v = b + lane;
      const uint32_t root = v < n ? p[v] : NONE;
      const uint32_t root0 = __shfl_sync(FULL, root, 0);
      // lanes under lane 0's root: lane 0 is the smallest of them
      if (v < n && (root != root0 || lane == 0) && (uint32_t)v < *(volatile uint32_t *)(rw + root))
        atomicMin(rw + root, (uint32_t)v);
    }
    asm volatile("bar.sync 1, %0;" ::"n"(NO) : "memory");
    for (int v = threadIdx.x; v < n; v += NO) {
      const uint32_t root = p[v], low = rw[root];
      A.labels[v0 + v] = (int32_t)min(low, root);
    }
  }
  if (A.mask) {
    uint8_t *mask = A.mask + e0;
    const int head = (int)((16 - (reinterpret_cast<uintptr_t>(mask) & 15)) & 15);
    const int h = head < m ? head : m, nq = (m - h) >> 4;
    uint4 *q = reinterpret_cast<uint4 *>(mask + h);
    for (int e = threadIdx.x; e < h; e += NO) mask[e] = (uint8_t)((bits[e >> 5] >> (e & 31)) & 1u);
    for (int i = threadIdx.x; i < nq; i += NO) q[i] = spread16(bits16(bits, h + ((int64_t)i << 4)));
    for (int e = h + (nq << 4) + threadIdx.x; e < m; e += NO) mask[e] = (uint8_t)((bits[e >> 5] >> (e & 31)) & 1u);
  }
}

constexpr size_t SMEM_MAX = 227 << 10;
constexpr size_t SMEM_STATIC = 13 << 10;  // sums, bins and the rest of a block's shared memory

template <int NT>
int launch_small(const SmallArgs &A, int blocks, size_t dyn, cudaStream_t s) {
  void (*fn)(SmallArgs) = A.wtype == MSF_F32 ? k_small<NT, true> : k_small<NT, false>;
  if (dyn + SMEM_STATIC > (48 << 10))
    MSF_CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(SMEM_MAX - SMEM_STATIC)));
  fn<<<blocks, NT, dyn, s>>>(A);
  return MSF_OK;
}

// Two side streams per device for launches that run beside each other: a
// branch starts after the work queued on the caller's stream and is waited for
// by it at the join.  Calls that share them only wait a little more.
struct Fork {
  cudaStream_t s;
  int n = 0;
  cudaStream_t used[2];
  explicit Fork(cudaStream_t st) : s(st) {}
  static int side(int i, cudaStream_t *out) {
    static std::mutex mu;
    static cudaStream_t streams[64][2] = {};
    int dev = 0;
    MSF_CK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(MSF_ERR_INVALID_ARG, "device ordinal out of range");
    std::lock_guard<std::mutex> lk(mu);
    if (!streams[dev][i]) MSF_CK(cudaStreamCreateWithFlags(&streams[dev][i], cudaStreamNonBlocking));
    *out = streams[dev][i];
    return MSF_OK;
  }
  // `to` waits for what is queued on `from`
  static int after(cudaStream_t from, cudaStream_t to) {
    cudaEvent_t ev;
    MSF_CK(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    cudaError_t e = cudaEventRecord(ev, from);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(to, ev, 0);
    cudaEventDestroy(ev);
    return e == cudaSuccess ? MSF_OK : cuda_fail(e, "ordering streams");
  }
  int branch() {
    if (int rc = side(n, &used[n])) return rc;
    return after(s, used[n++]);
  }
  int join() {
    int rc = MSF_OK;
    for (int i = 0; i < n; ++i)
      if (const int r = after(used[i], s)) {
        cudaStreamSynchronize(used[i]);  // (the blocks' memory is given back after this call)
        rc = r;
      }
    n = 0;
    return rc;
  }
};

}  // namespace

bool small_fits(int64_t n, int64_t m) {
  return n <= 65536 && m <= ((int64_t)1 << 19) && small_smem(n, m) + SMEM_STATIC <= SMEM_MAX;
}

// One block against solve.cu's grid: the block's passes and rounds grow with the
// edges and vertices, the grid's are a dozen barrier-bound phases.  Whole calls
// in us at (n, m), block / grid: (20000, 40000) 245 / 175, (14000, 131072) 229 / 186,
// (14000, 28000) 180 / 168, (10000, 40000) 134 / 170, (8000, 100000) 165 / 174, (8000,
// 200000) 219 / 178, (4000, 130000) 143 / 163, (4000, 400000) 276 / 162, (1000, 100000)
// 114 / 153.
bool small_single(int64_t n, int64_t m) { return small_fits(n, m) && m + 12 * n <= ((int64_t)11 << 14); }

// The same with the loop's rounds counted, which needs every edge in every round:
// (8000, 16000) 115 / 166, (1500, 15000) 109 / 147, (1500, 40000) 207 / 153,
// (8000, 60000) 345 / 195.
bool small_counted(int64_t n, int64_t m) { return small_fits(n, m) && m <= ((int64_t)3 << 13); }

// With `beside` the blocks are queued on a side stream that starts after the work
// queued on `s` so far.
int SmallRun::start(int32_t K, const int32_t *which, const int64_t *voff, const int64_t *eoff, const int32_t *src,
                    const int32_t *dst, const int2 *ends, const uint32_t *w, int wtype, uint8_t *mask, int32_t *labels,
                    double *totals, bool count, bool beside, cudaStream_t s) {
  const int64_t n = which ? 0 : voff[1], m = which ? 0 : eoff[1];
  const int32_t G = which ? K : 1;
  SmallArgs A;
  std::memset(&A, 0, sizeof(A));
  A.src = src;
  A.dst = dst;
  A.ends = ends;
  A.count = count;
  A.w = w;
  A.wtype = wtype;
  A.vec = ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(w)) & 15) == 0;
  A.n = n;
  A.m = m;
  A.mask = mask;
  A.labels = labels;
  A.totals = totals;
  int err = MSF_OK;
  // pinned: status words, then the offsets and the blocks' graphs, which the
  // blocks read in place (a copy would cost a call more than their one read)
  if (int rc = pin.take(64 + (which ? (size_t)K * SMALL_TABLE : 0))) return rc;
  A.host = pin.p;
  int64_t entries = m + 256;
  for (int32_t k = 0; which && k < K; ++k) entries += eoff[which[k] + 1] - eoff[which[k]] + 256;
  char *base = (char *)pool_alloc((size_t)entries * 16, &err);
  if (err) return err;
  list = base;
  stream = s;
  A.list = (uint4 *)base;
  int rc = MSF_OK;
  if (!which) {
    const size_t dyn = small_smem(n, m);
    rc = m <= 512 ? launch_small<256>(A, 1, dyn, s) : launch_small<1024>(A, 1, dyn, s);
  } else {
    // by block: vertex and edge offsets of its graph, its list, its number
    int64_t *hv = (int64_t *)(pin.p + 16), *he = hv + 2 * K, *hl = he + 2 * K;
    int32_t *order = (int32_t *)(hl + K);
    // graphs by falling size class
    int64_t count[42] = {0}, at[42], run = 0;
    size_t need[42] = {0};
    auto cls = [&](int32_t g) {
      const int64_t k = (eoff[g + 1] - eoff[g]) + (voff[g + 1] - voff[g]);
      int b = 0;
      while (((int64_t)1 << b) <= k) ++b;
      return b;
    };
    for (int32_t k = 0; k < K; ++k) {
      const int32_t g = which[k];
      const int c = cls(g);
      ++count[c];
      const size_t d = small_smem(voff[g + 1] - voff[g], eoff[g + 1] - eoff[g]);
      if (d > need[c]) need[c] = d;
    }
    for (int c = 41; c >= 0; --c) {
      at[c] = run;
      run += count[c];
    }
    for (int32_t k = 0; k < K; ++k) order[at[cls(which[k])]++] = which[k];
    int64_t entry = 0;
    for (int32_t k = 0; k < K; ++k) {
      const int32_t g = order[k];
      hv[2 * k] = voff[g];
      hv[2 * k + 1] = voff[g + 1];
      he[2 * k] = eoff[g];
      he[2 * k + 1] = eoff[g + 1];
      hl[k] = entry;
      entry += eoff[g + 1] - eoff[g] + 256;
    }
    // one launch per block size, side by side: 1024 threads (one block per SM)
    // for graphs from 2^13 vertices and edges on (for all while every graph
    // has an SM), 512 from 2^11 on, 256 below
    const bool few = G <= sm_count();
    const int from[3] = {few ? 0 : 14, 12, 0}, to[3] = {42, few ? 0 : 14, few ? 0 : 12};
    int64_t blocks[3] = {0, 0, 0};
    size_t dyn[3] = {0, 0, 0};
    int tiers = 0;
    for (int t = 0; t < 3; ++t) {
      for (int c = from[t]; c < to[t]; ++c) {
        blocks[t] += count[c];
        if (count[c] && need[c] > dyn[t]) dyn[t] = need[c];
      }
      tiers += blocks[t] > 0;
    }
    Fork fork(s);
    for (int i = beside ? 0 : 1; i < tiers && rc == MSF_OK; ++i) rc = fork.branch();
    int64_t first = 0;
    int used = beside ? 1 : 0;
    for (int t = 0; t < 3 && rc == MSF_OK; ++t) {
      if (blocks[t] == 0) continue;
      A.order = order + first;
      A.voff = hv + 2 * first;
      A.eoff = he + 2 * first;
      A.loff = hl + first;
      first += blocks[t];
      cudaStream_t st = used ? fork.used[used - 1] : s;
      ++used;
      rc = t == 0   ? launch_small<1024>(A, (int)blocks[t], dyn[t], st)
           : t == 1 ? launch_small<512>(A, (int)blocks[t], dyn[t], st)
                    : launch_small<256>(A, (int)blocks[t], dyn[t], st);
    }
    if (beside) {
      if (fork.n) side = fork.used[0];
    } else if (const int rj = fork.join()) {
      rc = rc ? rc : rj;
    }
  }
  queued = true;
  if (rc) return rc;
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? MSF_OK : cuda_fail(e, "forests of small graphs");
}

// (the side stream's work is waited for here: nothing of it is left when the call
// returns)
int SmallRun::finish(unsigned *status, LoopCounts *counts) {
  queued = false;
  cudaError_t e = side ? cudaStreamSynchronize(side) : cudaSuccess;
  const cudaError_t e2 = cudaStreamSynchronize(stream);
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) return cuda_fail(e, "forests of small graphs");
  const volatile unsigned *st = (volatile unsigned *)pin.p;
  if (st[0]) *status |= 1u;
  if (st[1]) *status |= 2u;
  if (counts) {
    counts->hooked = counts->passes = (int32_t)st[2];
    counts->left = st[3];
    counts->edges = st[4];
    counts->kernels = 1;
  }
  return MSF_OK;
}

SmallRun::~SmallRun() {
  if (queued) {  // (an error after the start: what is queued ends before its memory goes back)
    if (side) cudaStreamSynchronize(side);
    cudaStreamSynchronize(stream);
  }
  pool_free(list);
}

// Forests of one graph (which = NULL), or of K graphs that fit (small_fits),
// `which` of the graphs with the host offsets voff, eoff.  Synchronizes `s`;
// *status: 1 = index out of range, 2 = NaN weight.
int solve_small(int32_t K, const int32_t *which, const int64_t *voff, const int64_t *eoff, const int32_t *src,
                const int32_t *dst, const uint32_t *w, int wtype, uint8_t *mask, int32_t *labels, double *totals,
                unsigned *status, cudaStream_t s) {
  SmallRun run;
  const int rc = run.start(K, which, voff, eoff, src, dst, nullptr, w, wtype, mask, labels, totals, false, false, s);
  return rc ? rc : run.finish(status, nullptr);
}

int solve_small_pairs(int64_t n, int64_t m, const int2 *ends, const uint32_t *w, int wtype, uint8_t *mask,
                      int32_t *labels, double *totals, LoopCounts *counts, cudaStream_t s) {
  const int64_t voff[2] = {0, n}, eoff[2] = {0, m};
  unsigned status = 0;
  SmallRun run;
  const int rc = run.start(1, nullptr, voff, eoff, nullptr, nullptr, ends, w, wtype, mask, labels, totals, true, false, s);
  return rc ? rc : run.finish(&status, counts);
}

}  // namespace msf
