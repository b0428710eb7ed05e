// Forests from edge lists, without a CSR: of one list, of the larger graphs of a
// batch, and of a kept graph from the ends and weights that its handle holds.
//
// The strict order on (weight, edge index) makes the forest unique, so any exact
// method returns the round loop's mask, labels and total.  A CSR costs several
// passes over two records per edge and every round of the loop sweeps all of
// them; here the edges are read once or twice:
//
//   select   one pass validates the edges and keeps the light ones, in two
//            classes: about CLASS1 * n edges below a first threshold key, those
//            up to CLASS2 * n below a second (keys of a sample; all edges when
//            m is not much larger than n);
//   rounds   Boruvka rounds on the first class until no edge is left between
//            two components: every component's minimum edge by a minimum on
//            its 64-bit key word, then every edge that is the minimum of one
//            of its ends hooks that root onto the other (tie breaking as in
//            Algorithm 2), then the ends are relabelled to their roots and the
//            edges inside a component dropped; the same on what is left of the
//            second class;
//   filter   a second pass over the endpoints drops the edges inside a
//            component of the light forest (nearly all of the heavy ones) and
//            the rounds finish on the others.
//
// The lightest edge that leaves a component is in the forest (Sec. 2.3), and an
// edge inside a component of the lighter edges' forest is not, so every step
// is exact.
//
// Every warp owns pages of the edges and a list of the same capacity in the
// same pages: it fills, reads, relabels and compacts its own list in place, so
// the lists need no global counters and cannot overflow.
// The rounds kernel is cooperative, one block of 1024 threads per SM; its
// phases meet at a grid barrier (1 to 2 us, bounded wait), which costs less
// than the kernel boundaries and conditional nodes of a graph loop (about 60
// launches in the CSR path's small calls).  What bounds the steps: select and
// filter the instruction issue and DRAM (R-MAT 20: 43 and 58 us for 201 MB
// each, from pairs of ends 42 and 52), the minimum passes L1 wavefronts (two parents and two minima
// gathered per edge), late rounds the barriers.
//
// Measured on the whole call (build and round loop over the CSR before, this
// after): R-MAT 26 112 -> 21.9 ms, the 256^3 grid 9.9 -> 2.31 ms, R-MAT 20 1.75
// -> 0.455 ms, uniform n = 10^6, m = 16 n 2.6 -> 0.51 ms, R-MAT 16 0.47 -> 0.174
// ms, 4096 graphs of 38 M vertices 26.3 -> 5.84 ms.  Fractions around these when
// they were chosen (CLASS1 0.25 to 1, CLASS2 1.2 to 3): R-MAT 26 20.7 to 22.9 ms,
// the grid 2.3 to 4.4, uniform 0.52 to 0.70, R-MAT 20 0.48 to 0.54; a single light
// class of 1.5 n: 28.4, 3.2, 0.68 and 0.57 ms.
#include <cstring>

#include "exact.cuh"
#include "grid.cuh"
#include "internal.cuh"

namespace msf {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int ET = 1024;        // threads per block, one block per SM
constexpr int EW = ET / 32;     // warps per block
constexpr int SAMPLES = 1024;   // sampled weights for the thresholds
constexpr int VOTES = 128;      // sampled edge ends for the giant component
constexpr int TS_BITS = 11;     // slots of the block's table of minima
constexpr int TS = 1 << TS_BITS;
constexpr unsigned TABLE_HITS = 16;  // of a batch's 256 ends: below, the table is not worth its instructions
constexpr int HOPS = 16;        // hops of one settling pass
constexpr int SHORT_CHAIN = 8;  // hops through L1 before a chain counts as long
constexpr int ROUND_CAP = 64;   // Boruvka rounds at most (components at least halve)
constexpr uint32_t CAND = 0x80000000u;  // list entry may be a minimum of one of its ends
constexpr uint32_t LONG = 0x80000000u;  // listed root whose chain goes on
// Edges of the first class, and of both light classes, per vertex.
constexpr double CLASS1 = 0.75, CLASS2 = 1.5;
// The light edges form one class where a second one saves less than its rounds'
// barriers cost.  Calls in us, one class / two, uniform unless said: (300 000, 9 M)
// 329 / 339, R-MAT 18 of 8 M edges 261 / 273, an 80^3 lattice 293 / 312, 96^3 352 /
// 372, (500 000, 4 M) 347 / 331, (500 000, 16 M) 446 / 397, (700 000, 16 M) 502 / 431,
// (10^6, 2 M) 437 / 381, (2 * 10^6, 4 M) 632 / 522, a 140^3 lattice 632 / 595.
inline bool two_classes(int64_t n, int64_t m) {
  return n >= (int64_t)14 << 16 || (m >= (int64_t)1 << 22 && n >= (int64_t)3 << 17);
}
// With the loop's rounds counted: all edges in one class, whose rounds are the
// loop's, or classes and a replay of the rounds on the forest.  In us, one class /
// classes: R-MAT 16 of 2^20 edges 178 / 225, (200 000, 2^20) 297 / 349, a 96^3
// lattice 416 / 515, R-MAT 18 of 2^21 257 / 288, of 2^22 355 / 306; (100 000, 2^21)
// 395 / 336, (300 000, 3 M) 490 / 389, (10^6, 4 M) 677 / 577.  Trees and little more
// are counted directly whatever their size, as the replay's list is then nearly
// all of their edges: a path of 8 M vertices 1159 / 2443, (8 M, 8 M) 1212 / 1974,
// (8 M, 12 M) 1826 / 2222, (8 M, 16 M) 2499 / 2470, (8 M, 24 M) 3667 / 2564.
inline bool count_by_replay(int64_t n, int64_t m) {
  if (5 * m < 8 * n) return false;
  return m >= (int64_t)3 << 20 || (m >= (int64_t)3 << 19 && m >= 10 * n);
}
// Edges left from which a round's roots are settled in a step of their own:
// below, all of them are in flight at once (155 648 threads) and the minimum
// pass follows the chains itself, one barrier and about 5 us less per round
// (R-MAT 16: 257 -> 199 us).  A graph with few more edges than vertices may be one
// long chain, whose edges all wait at the same parents: there from 2^15 on (a path
// with rising weights and permuted ids, 40 000 vertices 177 -> 140 us, 131 000
// 224 -> 155; for all graphs that line took R-MAT 16 from 174 to 184).
constexpr unsigned long long SMALL = 1 << 17, SMALL_CHAINS = 1 << 15;
// Edges or vertices per block of a call that does not fill the device.  (1024 a
// block take all SMs from 152 000 on and are no faster: 209 us against 205 at
// 30 000 vertices and 200 000 edges; 8192 251.)
constexpr int64_t BLOCK_SHARE = 4096;

constexpr size_t SMEM_BITS = 224 << 10;  // largest bitmap kept in shared memory

struct Ctrl {
  unsigned long long arrive[3][2];  // grid barriers of the rounds kernels
  unsigned abort;      // a barrier wait ran out
  unsigned err;        // 1 = index out of range, 2 = NaN weight
  unsigned pairs[4];   // trees formed, by round modulo 4
  unsigned edges;      // forest edges
  unsigned long long thresh[2];  // keys of the first class lie below [0], of the second below [1]
};

struct Args {
  int64_t n, m;
  const int32_t *src, *dst;
  const int2 *ends;     // instead of src and dst: validated ends
  const uint32_t *w;
  int32_t wtype;
  int32_t classes;      // 1 = every edge in the first class, 2 = none heavy, 3
  int32_t second;       // there is a second class
  int32_t smem_bits;    // the giant component's bitmap fits in shared memory
  int32_t es, vs;       // pages of 2^es edges and 2^vs vertices (see Pages)
  unsigned rank[2];     // the thresholds' ranks among SAMPLES
  int32_t *p;
  unsigned long long *r;
  int32_t *roots;       // per warp region: roots that may have edges
  uint32_t *gbits;      // vertices of the giant component, as a bitmap
  unsigned *front, *back;  // per warp: entries of the first and second class
  uint4 *list;          // (u, v, edge id, ordered weight), u | CAND
  uint32_t *mbits;
  // a batch (see Batch below); G = 0: one graph
  int32_t G;
  const int64_t *eL, *vL;  // [G + 1] first edge and vertex of each graph here
  const int64_t *eA, *vA;  // [G] first edge and vertex of each graph in the call's arrays
  const int32_t *id;       // [G] graph of the call
  int32_t *eg, *vg;        // graph of each page's first edge and first vertex
  int32_t *giant;          // [G] root of each graph's giant component
  unsigned long long *bins;  // [256] long accumulators (zeroed with the control block), [G][256] for a batch
  Ctrl *ctl;
  uint8_t *mask;
  int32_t *labels;
  double *totals;
  unsigned *host;       // pinned: [0] status bits, [1..4] rounds with hooks, trees the last left, edges, passes
};

__device__ __forceinline__ unsigned long long ld_rel64(const unsigned long long *a) {
  return cuda::atomic_ref<unsigned long long, cuda::thread_scope_device>(*const_cast<unsigned long long *>(a))
      .load(cuda::memory_order_relaxed);
}

// Root of x, whose parent y was read, by its chain.  Hooks happen in other
// phases, so the roots do not change meanwhile, and a parent read from L1 is an
// ancestor even when it is out of date.  Short chains are left as they are (a
// hub's many edges would all write its parent: 300 us of one pass over 88 000
// edges); a long one goes on in L2, is halved for the threads behind, and x
// then points to the root.
__device__ __forceinline__ int32_t chase(int32_t *p, int32_t x, int32_t y) {
  if (y == x) return x;
  const int32_t x0 = x;
  x = y;
  y = __ldca(p + x);
#pragma unroll 1
  for (int k = 0; k < SHORT_CHAIN && y != x; ++k) {
    x = y;
    y = __ldca(p + x);
  }
  if (y == x) return x;
  while (y != x) {
    const int32_t z = ld_rel(p + y);
    if (z != y) st_rel(p + x, z);
    x = z;
    y = ld_rel(p + x);
  }
  st_rel(p + x0, x);
  return x;
}

// The block's shared-memory table of minima.  A slot belongs to the first root
// that hashes to it; other roots go to r directly.  Late rounds have few
// roots, most edges end in one of them, and both its atomics and its reads
// would queue at one L2 line (R-MAT 20: 380 us for a pass over 1.2 M edges).
struct Table {
  int32_t key[TS];
  unsigned long long val[TS];
};
__device__ __forceinline__ void table_clear(Table &t) {
  for (int i = threadIdx.x; i < TS; i += ET) {
    t.key[i] = -1;
    t.val[i] = KEY_INF;
  }
}
// The table's slot for a root, or -1 when another root holds it; `hit`: the
// root held it already.
__device__ __forceinline__ int table_slot(Table &t, int32_t root, bool &hit) {
  const int slot = (int)(((uint32_t)root * 0x9E3779B1u) >> (32 - TS_BITS));
  int k = *(volatile int32_t *)(t.key + slot);
  hit = k == root;
  if (k == -1) {
    k = atomicCAS(t.key + slot, -1, root);
    if (k == -1) k = root;
  }
  return k == root ? slot : -1;
}
// Lowers the slot's minimum to `key`; whether it did.
__device__ __forceinline__ bool table_offer(Table &t, int slot, unsigned long long key) {
  unsigned long long old = *(volatile unsigned long long *)(t.val + slot);
  while (key < old) {
    const unsigned long long seen = atomicCAS(t.val + slot, old, key);
    if (seen == old) return true;
    old = seen;
  }
  return false;
}

// Minimum pass over `cnt` entries of the warp's list from place `from` on,
// which end up at its front: with RELABEL the ends become their roots first
// (their parents) and the entries inside a component are dropped.  Every end's
// minimum is lowered to the entry's key; it is read first, and only an entry
// that was below it is marked CAND (the final minimum is; lowering them unread
// took R-MAT 26 from 23 to 31 ms).  A warp leaves the block's table alone once
// few of its ends are found there (many small graphs: 9.0 -> 8.6 ms).  Returns
// the entries left.
template <bool RELABEL, bool CHASE>
__device__ __noinline__ unsigned min_pass(const Args &A, Table &tab, const Pages P, unsigned from, unsigned cnt) {
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  constexpr int U = 4;
  unsigned out = 0;
  bool use = true;
  for (unsigned b0 = 0; b0 < cnt; b0 += 32 * U) {
    uint4 x[U];
    bool on[U];
    int32_t u[U], v[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const unsigned i = b0 + j * 32 + lane;
      on[j] = i < cnt;
      x[j] = on[j] ? A.list[P.at(from + i)] : make_uint4(0u, 0u, 0u, 0u);
      u[j] = (int32_t)(x[j].x & ~CAND);
      v[j] = (int32_t)x[j].y;
    }
    if (RELABEL) {
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const int32_t a = u[j], b = v[j];
        u[j] = on[j] ? __ldca(A.p + a) : 0;
        v[j] = on[j] ? __ldca(A.p + b) : 0;
      }
      if (CHASE) {
#pragma unroll
        for (int j = 0; j < U; ++j) {
          if (!on[j]) continue;
          u[j] = chase(A.p, (int32_t)(x[j].x & ~CAND), u[j]);
          v[j] = chase(A.p, (int32_t)x[j].y, v[j]);
        }
      }
#pragma unroll
      for (int j = 0; j < U; ++j) on[j] = on[j] && u[j] != v[j];
    }
    unsigned cand = 0u;
    unsigned gu = 0, gv = 0;  // entries whose ends go to r directly
    if (use) {
      unsigned hits = 0;
#pragma unroll
      for (int j = 0; j < U; ++j) {
        if (!on[j]) continue;
        const unsigned long long key = ((unsigned long long)x[j].w << 32) | x[j].z;
        bool hu, hv;
        const int su = table_slot(tab, u[j], hu), sv = table_slot(tab, v[j], hv);
        hits += (hu ? 1u : 0u) + (hv ? 1u : 0u);
        if (su < 0) gu |= 1u << j;
        else if (table_offer(tab, su, key)) cand |= 1u << j;
        if (sv < 0) gv |= 1u << j;
        else if (table_offer(tab, sv, key)) cand |= 1u << j;
      }
      use = __reduce_add_sync(FULL, hits) >= TABLE_HITS;
    } else {
#pragma unroll
      for (int j = 0; j < U; ++j)
        if (on[j]) gu |= 1u << j;
      gv = gu;
    }
    {
      unsigned long long ru[U], rv[U];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        ru[j] = gu >> j & 1u ? ld_rel64(A.r + u[j]) : 0ull;
        rv[j] = gv >> j & 1u ? ld_rel64(A.r + v[j]) : 0ull;
      }
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const unsigned long long key = ((unsigned long long)x[j].w << 32) | x[j].z;
        if (key >= ru[j]) gu &= ~(1u << j);
        if (key >= rv[j]) gv &= ~(1u << j);
      }
      cand |= gu | gv;
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const unsigned long long key = ((unsigned long long)x[j].w << 32) | x[j].z;
      if (gu >> j & 1u) atomicMin(A.r + u[j], key);
      if (gv >> j & 1u) atomicMin(A.r + v[j], key);
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const unsigned bal = __ballot_sync(FULL, on[j]);
      const unsigned at = out + __popc(bal & below);
      if (on[j])
        A.list[P.at(at)] = make_uint4((uint32_t)u[j] | (cand >> j & 1u ? CAND : 0u), (uint32_t)v[j], x[j].z, x[j].w);
      out += __popc(bal);
    }
  }
  __syncwarp();
  return out;
}

// Hooks along every entry that is the minimum of one of its ends (tie
// breaking: of two roots that chose the same edge the smaller stays a root).
// Returns the hooks of the thread in the low half and those of two roots that
// chose each other, one for every tree formed, in the high half.
__device__ __noinline__ unsigned hook_pass(const Args &A, const Pages P, unsigned cnt, bool small, bool mark, bool sum,
                                           BlockSums &sums, unsigned long long &usum) {
  const int lane = threadIdx.x & 31;
  constexpr int U = 4;
  unsigned hooks = 0;
  for (unsigned b0 = 0; b0 < cnt; b0 += 32 * U) {
    uint4 x[U];
    unsigned long long ru[U], rv[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const unsigned i = b0 + j * 32 + lane;
      x[j] = i < cnt ? A.list[P.at(i)] : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const bool c = (x[j].x & CAND) != 0;
      ru[j] = c ? __ldca(A.r + (x[j].x & ~CAND)) : KEY_INF;
      rv[j] = c ? __ldca(A.r + x[j].y) : KEY_INF;
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int32_t u = (int32_t)(x[j].x & ~CAND), v = (int32_t)x[j].y;
      const unsigned long long key = ((unsigned long long)x[j].w << 32) | x[j].z;
      const bool mu = ru[j] == key, mv = rv[j] == key;
      if (!((x[j].x & CAND) && (mu || mv))) continue;
      hooks += mu && mv ? 0x10001u : 1u;
      if (small) {  // the minima are cleared here (no other entry's key equals them, before or after)
        if (mu) A.r[u] = KEY_INF;
        if (mv) A.r[v] = KEY_INF;
      }
      if (mu && (!mv || v < u)) A.p[u] = v;
      else A.p[v] = u;
      if (mark) atomicOr(A.mbits + (x[j].z >> 5), 1u << (x[j].z & 31u));
      if (sum) {
        if (A.wtype == MSF_U32) usum += x[j].w;
        else sums.add(x[j].w);
      }
    }
  }
  return hooks;
}

// A batch of graphs is solved as one graph whose edges and vertices are those
// of its graphs, one after the other (eL, vL): positions there index parents,
// lists and the bitmap, and order the edges of a graph as their own indices
// do.  A page of edges meets one or a few graphs; `f(g, x, k)` gets each piece
// of the page's: graph g, its first position x and its k edges.
template <class F>
__device__ __forceinline__ void for_pieces(const Args &A, uint32_t page, F f) {
  const int64_t lo = (int64_t)page << A.es, full = lo + ((int64_t)1 << A.es), hi = full < A.m ? full : A.m;
  int g = A.eg[page];
  for (int64_t x = lo; x < hi; ++g) {
    const int64_t end = A.eL[g + 1] < hi ? A.eL[g + 1] : hi;
    if (end > x) f(g, x, (int)(end - x));
    x = end;
  }
}
// graph of vertex v, from a graph that is not behind it
__device__ __forceinline__ int graph_from(const Args &A, int g, int64_t v) {
  while (g + 1 < A.G && A.vL[g + 1] <= v) ++g;
  return g;
}
// graph of position x, off[g] <= x < off[g + 1]
__device__ __forceinline__ int graph_at(const int64_t *off, int G, int64_t x) {
  int a = 0, b = G;
  while (b - a > 1) {
    const int mid = (a + b) >> 1;
    if (off[mid] <= x) a = mid;
    else b = mid;
  }
  return a;
}

// Four consecutive edges of a lane.
struct Quad {
  int4 s, d;
  uint4 w;
};
// Forms of the edges: separate arrays of ends, aligned or not, or pairs.
enum Form { SCALAR = 0, VECTOR = 1, PAIRS = 2 };
template <int FORM>
__device__ __forceinline__ Quad load_quad(const Args &A, int64_t e, int64_t hi) {
  Quad q;
  q.s = q.d = make_int4(0, 0, 0, 0);
  q.w = make_uint4(0u, 0u, 0u, 0u);
  if (FORM == PAIRS) {
    load_pairs(A.ends, e, hi, q.s, q.d);
    uint32_t *w = &q.w.x;
    if (e + 4 <= hi) q.w = __ldcs(reinterpret_cast<const uint4 *>(A.w + e));
    else
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (e + j < hi) w[j] = A.w[e + j];
  } else if (FORM == VECTOR && e + 4 <= hi) {
    q.s = __ldcs(reinterpret_cast<const int4 *>(A.src + e));
    q.d = __ldcs(reinterpret_cast<const int4 *>(A.dst + e));
    q.w = __ldcs(reinterpret_cast<const uint4 *>(A.w + e));
  } else if (e < hi) {
    q.s.x = A.src[e];
    q.d.x = A.dst[e];
    q.w.x = A.w[e];
    if (e + 1 < hi) {
      q.s.y = A.src[e + 1];
      q.d.y = A.dst[e + 1];
      q.w.y = A.w[e + 1];
    }
    if (e + 2 < hi) {
      q.s.z = A.src[e + 2];
      q.d.z = A.dst[e + 2];
      q.w.z = A.w[e + 2];
    }
    if (e + 3 < hi) {
      q.s.w = A.src[e + 3];
      q.d.w = A.dst[e + 3];
      q.w.w = A.w[e + 3];
    }
  }
  return q;
}

// Their ends only.
struct Ends {
  int4 s, d;
};
template <int FORM>
__device__ __forceinline__ Ends load_ends(const Args &A, int64_t e, int64_t hi) {
  Ends q;
  q.s = q.d = make_int4(0, 0, 0, 0);
  if (FORM == PAIRS) {
    load_pairs(A.ends, e, hi, q.s, q.d);
  } else if (FORM == VECTOR && e + 4 <= hi) {
    q.s = __ldcs(reinterpret_cast<const int4 *>(A.src + e));
    q.d = __ldcs(reinterpret_cast<const int4 *>(A.dst + e));
  } else if (e < hi) {
    int32_t *s = &q.s.x, *d = &q.d.x;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (e + j < hi) {
        s[j] = A.src[e + j];
        d[j] = A.dst[e + j];
      }
  }
  return q;
}

// First pass over the warp's edges: validation; the non-loop edges below T0 go
// to the front of the warp's list, those from T0 to T1 to its back (growing
// downwards from its end).  The pass is bound by instruction issue, so an edge costs a
// running maximum (the index check), a NaN test and one or two comparisons
// until it is selected.
template <int FORM, bool F32>
__device__ __forceinline__ void select_pass(const Args &A, const Pages P, unsigned long long T0,
                                            unsigned long long T1, unsigned &front, unsigned &back, unsigned &err) {
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  const uint32_t n = (uint32_t)A.n;
  front = back = err = 0;
  if (!P.cap) return;
  const unsigned last = P.cap - 1u;
  Limit<F32> l0(T0), l1(T1);
  uint32_t top = 0;  // largest index seen
  bool nan = false;
  // (zeros past the end: self-loops)
  auto load = [&](int b) { return load_quad<FORM>(A, P.at((uint32_t)b) + 4 * lane, (uint32_t)b < P.cap ? A.m : 0); };
  auto body = [&](const Quad &q, int i) {
    const int64_t b = P.at((uint32_t)i), e0 = b + 4 * lane;
    const uint32_t u[4] = {(uint32_t)q.s.x, (uint32_t)q.s.y, (uint32_t)q.s.z, (uint32_t)q.s.w};
    const uint32_t v[4] = {(uint32_t)q.d.x, (uint32_t)q.d.y, (uint32_t)q.d.z, (uint32_t)q.d.w};
    const uint32_t w[4] = {q.w.x, q.w.y, q.w.z, q.w.w};
    l0.batch(b);
    l1.batch(b);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (FORM != PAIRS) {
        top = max(top, max(u[j], v[j]));
        if (F32) nan |= __uint_as_float(w[j]) != __uint_as_float(w[j]);
      }
      const bool sel = l1.below(w[j]) && u[j] != v[j];
      const unsigned m = __ballot_sync(FULL, sel);
      if (!m) continue;
      // (an edge with an invalid index is selected too; it is never used)
      const unsigned mf = __ballot_sync(FULL, sel && l0.below(w[j]));
      const bool fr = mf >> lane & 1u;
      if (sel) {
        const unsigned at = fr ? front + __popc(mf & below) : last - (back + __popc(m & ~mf & below));
        A.list[P.at(at)] = make_uint4(u[j], v[j], (uint32_t)(e0 + j), ord_weight_dev(w[j], F32 ? MSF_F32 : MSF_U32));
      }
      front += __popc(mf);
      back += __popc(m & ~mf);
    }
  };
  stream2<Quad>(0, (int)P.cap, load, body);
  if (FORM != PAIRS) err = (top >= n ? 1u : 0u) | (nan ? 2u : 0u);
  __syncwarp();
}

// Second pass over the warp's edges: those whose ends lie in different
// components go to the list, as roots (parents are roots here).  A light edge
// lies inside a component, so the weights are read for the edges left only.
// Most edges lie inside the giant component: two bits of its bitmap tell,
// from shared memory when it fits there (a gather of parents is one L1
// wavefront per lane; R-MAT 20: 30 M of them).
template <int FORM, bool SMEM>
__device__ __forceinline__ unsigned filter_pass(const Args &A, const Pages P, const uint32_t *bits) {
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  unsigned out = 0;
  // (zeros past the end: self-loops)
  auto load = [&](int b) { return load_ends<FORM>(A, P.at((uint32_t)b) + 4 * lane, (uint32_t)b < P.cap ? A.m : 0); };
  auto body = [&](const Ends &q, int i) {
    const int64_t e0 = P.at((uint32_t)i) + 4 * lane, hi = A.m;
    int32_t u[4] = {q.s.x, q.s.y, q.s.z, q.s.w}, v[4] = {q.d.x, q.d.y, q.d.z, q.d.w};
    uint32_t bu[4], bv[4], w[4];
    bool on[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      bu[j] = SMEM ? bits[(uint32_t)u[j] >> 5] : __ldca(bits + ((uint32_t)u[j] >> 5));
      bv[j] = SMEM ? bits[(uint32_t)v[j] >> 5] : __ldca(bits + ((uint32_t)v[j] >> 5));
    }
    bool any = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      on[j] = !(__funnelshift_r(bu[j], bu[j], u[j]) & __funnelshift_r(bv[j], bv[j], v[j]) & 1u);
      any |= on[j];
    }
    if (!__any_sync(FULL, any)) return;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      on[j] = on[j] && e0 + j < hi;
      w[j] = on[j] ? __ldcs(A.w + e0 + j) : 0u;
      u[j] = on[j] ? __ldca(A.p + u[j]) : 0;
      v[j] = on[j] ? __ldca(A.p + v[j]) : 0;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool o = u[j] != v[j];
      const unsigned bal = __ballot_sync(FULL, o);
      if (o)
        A.list[P.at(out + __popc(bal & below))] =
            make_uint4((uint32_t)u[j], (uint32_t)v[j], (uint32_t)(e0 + j), ord_weight_dev(w[j], A.wtype));
      out += __popc(bal);
    }
  };
  stream2<Ends>(0, (int)P.cap, load, body);
  __syncwarp();
  return out;
}

// The same passes over a batch, piece by piece (the thresholds' edge indices
// are positions, compared edge by edge).
template <bool F32>
__device__ __forceinline__ void select_batch(const Args &A, bool vec, const Pages P, unsigned long long T0,
                                             unsigned long long T1, unsigned &front, unsigned &back, unsigned &err) {
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  front = back = 0;
  const unsigned last = P.cap - 1u;
  Limit<F32> l0(T0), l1(T1);
  bool bad = false, nan = false;
  auto piece = [&](int g, int64_t x, int k) {
    const int64_t a = A.eA[g] + (x - A.eL[g]), base = a & ~(int64_t)3;
    const uint32_t vb = (uint32_t)A.vL[g], lim = (uint32_t)(A.vL[g + 1] - A.vL[g]);
    const int first = (int)(a - base), end = first + k;
    const int32_t *S = A.src + base, *D = A.dst + base;
    const uint32_t *W = A.w + base;
    auto load = [&](int b) { return edge_quad<true>(S, D, W, vec, b + 4 * lane, first, end); };
    auto body = [&](const EdgeQuad &q, int b) {
      const int i = b + 4 * lane;
      const uint32_t u[4] = {(uint32_t)q.s.x, (uint32_t)q.s.y, (uint32_t)q.s.z, (uint32_t)q.s.w};
      const uint32_t v[4] = {(uint32_t)q.d.x, (uint32_t)q.d.y, (uint32_t)q.d.z, (uint32_t)q.d.w};
      const uint32_t w[4] = {q.w.x, q.w.y, q.w.z, q.w.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t e = x + (i + j - first);
        bad |= max(u[j], v[j]) >= lim;
        if (F32) nan |= __uint_as_float(w[j]) != __uint_as_float(w[j]);
        const bool sel = u[j] != v[j] && l1.below(w[j], e);
        const unsigned m = __ballot_sync(FULL, sel);
        if (!m) continue;
        const unsigned mf = __ballot_sync(FULL, sel && l0.below(w[j], e));
        const bool fr = mf >> lane & 1u;
        if (sel) {
          const unsigned at = fr ? front + __popc(mf & below) : last - (back + __popc(m & ~mf & below));
          A.list[P.at(at)] = make_uint4(u[j] + vb, v[j] + vb, (uint32_t)e, ord_weight_dev(w[j], F32 ? MSF_F32 : MSF_U32));
        }
        front += __popc(mf);
        back += __popc(m & ~mf);
      }
    };
    stream2<EdgeQuad>(0, end, load, body);
  };
  for (uint32_t i = 0; i < P.cap; i += 1u << P.s) for_pieces(A, P.page(i), piece);
  err = (bad ? 1u : 0u) | (nan ? 2u : 0u);
  __syncwarp();
}

template <bool SMEM>
__device__ __forceinline__ unsigned filter_batch(const Args &A, bool vec, const Pages P, const uint32_t *bits) {
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  unsigned out = 0;
  auto piece = [&](int g, int64_t x, int k) {
    const int64_t a = A.eA[g] + (x - A.eL[g]), base = a & ~(int64_t)3;
    const int32_t vb = (int32_t)A.vL[g];
    const int first = (int)(a - base), end = first + k;
    const int32_t *S = A.src + base, *D = A.dst + base;
    const uint32_t *W = A.w + base;
    auto load = [&](int b) { return edge_quad<false>(S, D, W, vec, b + 4 * lane, first, end); };
    auto body = [&](const EdgeQuad &q, int b) {
      const int i = b + 4 * lane;
      int32_t u[4] = {q.s.x + vb, q.s.y + vb, q.s.z + vb, q.s.w + vb};
      int32_t v[4] = {q.d.x + vb, q.d.y + vb, q.d.z + vb, q.d.w + vb};
      uint32_t w[4];
      bool on[4], any = false;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t bu = SMEM ? bits[u[j] >> 5] : __ldca(bits + (u[j] >> 5));
        const uint32_t bv = SMEM ? bits[v[j] >> 5] : __ldca(bits + (v[j] >> 5));
        on[j] = u[j] != v[j] && !(__funnelshift_r(bu, bu, u[j]) & __funnelshift_r(bv, bv, v[j]) & 1u);
        any |= on[j];
      }
      if (!__any_sync(FULL, any)) return;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        w[j] = on[j] ? __ldcs(W + i + j) : 0u;
        u[j] = on[j] ? __ldca(A.p + u[j]) : 0;
        v[j] = on[j] ? __ldca(A.p + v[j]) : 0;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool o = u[j] != v[j];
        const unsigned bal = __ballot_sync(FULL, o);
        if (o)
          A.list[P.at(out + __popc(bal & below))] = make_uint4(
              (uint32_t)u[j], (uint32_t)v[j], (uint32_t)(x + (i + j - first)), ord_weight_dev(w[j], A.wtype));
        out += __popc(bal);
      }
    };
    stream2<EdgeQuad>(0, end, load, body);
  };
  for (uint32_t i = 0; i < P.cap; i += 1u << P.s) for_pieces(A, P.page(i), piece);
  __syncwarp();
  return out;
}

// The thresholds: the sample's keys (edge indices rounded down to a batch) of the two wanted ranks, found bit by bit
// (one sample per thread, block 0).  The low half of a key, the edge index,
// only matters where many samples share the threshold's weight.
__device__ void pick_thresholds(const Args &A) {
  static_assert(SAMPLES == ET, "one sample per thread");
  const int64_t step = A.m / SAMPLES;  // m >= SAMPLES
  const int64_t i = threadIdx.x;
  const uint32_t h = (uint32_t)i * 0x9E3779B1u;
  const int64_t e = i * A.m / SAMPLES + (int64_t)(((uint64_t)h * (uint64_t)step) >> 32);
  int64_t ea = e;
  if (A.G) {
    const int g = graph_at(A.eL, A.G, e);
    ea = A.eA[g] + (e - A.eL[g]);
  }
  const uint32_t w = ord_weight_dev(A.w[ea], A.wtype);
  const unsigned r0 = A.rank[0], r1 = A.rank[1];
  uint32_t w0 = 0, w1 = 0;
  for (int b = 31; b >= 0; --b) {
    const uint32_t c0 = w0 | (1u << b), c1 = w1 | (1u << b);
    if (__syncthreads_count(w < c0) <= (int)r0) w0 = c0;
    if (__syncthreads_count(w < c1) <= (int)r1) w1 = c1;
  }
  // samples below w0: at most r0; with those equal to it: more
  uint32_t e0 = 0xffffffffu, e1 = 0xffffffffu;
  if (__syncthreads_count(w <= w0) > (int)(r0 + r0 / 4 + 1) || __syncthreads_count(w <= w1) > (int)(r1 + r1 / 4 + 1)) {
    e0 = e1 = 0;
    for (int b = 31; b >= 0; --b) {
      const uint32_t c0 = e0 | (1u << b), c1 = e1 | (1u << b);
      if (__syncthreads_count(w < w0 || (w == w0 && (uint32_t)e < c0)) <= (int)r0) e0 = c0;
      if (__syncthreads_count(w < w1 || (w == w1 && (uint32_t)e < c1)) <= (int)r1) e1 = c1;
    }
  }
  if (threadIdx.x == 0) {
    A.ctl->thresh[0] = ((unsigned long long)w0 << 32) | (e0 == 0xffffffffu ? e0 : e0 & ~127u);
    A.ctl->thresh[1] = ((unsigned long long)w1 << 32) | (e1 == 0xffffffffu ? e1 : e1 & ~127u);
  }
}

// The root that most of VOTES sampled edge ends lie under (every block finds
// the same one): the giant component, when there is one.
__device__ int32_t vote_giant(const Args &A) {
  __shared__ int32_t vote[VOTES];
  __shared__ unsigned best;
  if (threadIdx.x == 0) best = 0;
  if (threadIdx.x < VOTES) {
    const int64_t e = (int64_t)((unsigned long long)threadIdx.x * (unsigned long long)A.m / VOTES);
    int32_t x = A.ends ? ((threadIdx.x & 1) ? A.ends[e].x : A.ends[e].y) : (threadIdx.x & 1) ? A.src[e] : A.dst[e];
    if ((uint32_t)x >= (uint32_t)A.n) x = 0;  // (an invalid edge: the call fails later)
    int32_t y = __ldca(A.p + x);
    while (y != x) {
      x = y;
      y = __ldca(A.p + x);
    }
    vote[threadIdx.x] = x;
  }
  __syncthreads();
  if (threadIdx.x < VOTES) {
    unsigned c = 0;
    for (int i = 0; i < VOTES; ++i) c += vote[i] == vote[threadIdx.x];
    atomicMax(&best, (c << 16) | (unsigned)threadIdx.x);
  }
  __syncthreads();
  return vote[best & 0xffffu];
}

// The same for every graph of a batch, a warp each (32 sampled ends).
__device__ void vote_giants(const Args &A, int64_t warp, int64_t nwarps) {
  const int lane = threadIdx.x & 31;
  for (int64_t g = warp; g < A.G; g += nwarps) {
    const int64_t k = A.eL[g + 1] - A.eL[g], e = A.eA[g] + (int64_t)lane * k / 32;
    int32_t x = -1;
    if (k > 0) {
      x = (int32_t)A.vL[g] + ((lane & 1) ? A.src[e] : A.dst[e]);
      int32_t y = __ldca(A.p + x);
      while (y != x) {
        x = y;
        y = __ldca(A.p + x);
      }
    }
    const unsigned best = __reduce_max_sync(FULL, ((unsigned)__popc(__match_any_sync(FULL, x)) << 8) | (unsigned)lane);
    x = __shfl_sync(FULL, x, (int)(best & 31u));
    if (lane == 0) A.giant[g] = x;
  }
}

// Parents, minima, root lists and the forest bitmap; the thresholds.
__global__ void __launch_bounds__(ET, 1) k_prepare(Args A) {
  const int64_t tid = (int64_t)blockIdx.x * ET + threadIdx.x, nthr = (int64_t)gridDim.x * ET;
  for (int64_t v = tid; v < A.n; v += nthr) {
    A.p[v] = (int32_t)v;
    A.r[v] = KEY_INF;
    A.roots[v] = (int32_t)v;
  }
  if (A.mbits) {
    const int64_t words = (A.m + 31) / 32 + 2;
    for (int64_t i = tid; i < words; i += nthr) A.mbits[i] = 0u;
  }
  if (A.G) {
    for (int64_t i = tid; i < (int64_t)A.G * 256; i += nthr) A.bins[i] = 0ull;
    for (int64_t i = tid; i << A.es < A.m; i += nthr) A.eg[i] = graph_at(A.eL, A.G, i << A.es);
    for (int64_t i = tid; i << A.vs < A.n; i += nthr) A.vg[i] = graph_at(A.vL, A.G, i << A.vs);
  }
  if (A.classes > 1 && blockIdx.x == 0) pick_thresholds(A);
}

template <int FORM, bool F32, bool BATCH>
__global__ void __launch_bounds__(ET, 1) k_select(Args A) {
  const int64_t warp = ((int64_t)blockIdx.x * ET + threadIdx.x) >> 5;
  const Pages P(A.m, A.es, warp, (int64_t)gridDim.x * EW);
  const unsigned long long T0 = A.classes > 1 ? A.ctl->thresh[0] : KEY_INF;
  const unsigned long long T1 = A.classes > 2 ? A.ctl->thresh[1] : KEY_INF;
  unsigned front, back, err = 0;
  if (BATCH) select_batch<F32>(A, FORM == VECTOR, P, T0, T1, front, back, err);
  else select_pass<FORM, F32>(A, P, T0, T1, front, back, err);
  if (err) atomicOr(&A.ctl->err, err);
  if ((threadIdx.x & 31) == 0) {  // (an invalid edge ends the call: no list is used)
    A.front[warp] = front;
    A.back[warp] = back;
  }
}

template <int FORM, bool SMEM, bool BATCH>
__global__ void __launch_bounds__(ET, 1) k_filter(Args A) {
  extern __shared__ uint32_t dyn_bits[];
  const int64_t warp = ((int64_t)blockIdx.x * ET + threadIdx.x) >> 5;
  const Pages P(A.m, A.es, warp, (int64_t)gridDim.x * EW);
  unsigned front = 0;
  if (!A.ctl->err && !A.ctl->abort) {  // (an invalid edge's index must not be used)
    if (SMEM) {
      const int64_t words = (A.n + 31) / 32;
      for (int64_t i = threadIdx.x; i < words; i += ET) dyn_bits[i] = A.gbits[i];
      __syncthreads();
    }
    const uint32_t *bits = SMEM ? dyn_bits : A.gbits;
    front = BATCH ? filter_batch<SMEM>(A, FORM == VECTOR, P, bits) : filter_pass<FORM, SMEM>(A, P, bits);
  }
  if ((threadIdx.x & 31) == 0) A.front[warp] = front;
}

// Mask bytes of the warp's positions of a batch, and the weights of the
// forest edges among them into their graphs' accumulators: a piece's sums of
// four exponents from its first forest weight's down are kept in registers.
__device__ void batch_results(const Args &A, const Pages P) {
  const int lane = threadIdx.x & 31;
  constexpr int WIN = 4, U = 4;
  auto piece = [&](int g, int64_t x, int k) {
    const int64_t a = A.eA[g] + (x - A.eL[g]);
    if (A.mask) {
      uint8_t *mask = A.mask + a;
      const int head = (int)((16 - (reinterpret_cast<uintptr_t>(mask) & 15)) & 15);
      const int h = head < k ? head : k, nq = (k - h) >> 4;
      uint4 *q = reinterpret_cast<uint4 *>(mask + h);
      auto bit = [&](int i) { return (uint8_t)((A.mbits[(x + i) >> 5] >> ((x + i) & 31)) & 1u); };
      for (int i = lane; i < h; i += 32) mask[i] = bit(i);
      for (int i = lane; i < nq; i += 32) q[i] = spread16(bits16(A.mbits, x + h + ((int64_t)i << 4)));
      for (int i = h + (nq << 4) + lane; i < k; i += 32) mask[i] = bit(i);
    }
    if (!A.totals) return;
    const uint32_t *W = A.w + a;
    unsigned long long *bins = A.bins + (int64_t)g * 256;
    long long acc[WIN];
#pragma unroll
    for (int i = 0; i < WIN; ++i) acc[i] = 0;
    int top = -1;
    for (int b0 = 0; b0 < k; b0 += 32 * U) {
      bool on[U];
      uint32_t w[U];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const int i = b0 + j * 32 + lane;
        on[j] = i < k && ((A.mbits[(x + i) >> 5] >> ((x + i) & 31)) & 1u);
        w[j] = on[j] ? W[i] : 0u;
      }
#pragma unroll
      for (int j = 0; j < U; ++j) {
        int bin = 0;
        long long val = 0;
        if (on[j]) weight_bin(ord_weight_dev(w[j], A.wtype), A.wtype, &bin, &val);
        if (top < 0 && __any_sync(FULL, on[j])) top = __reduce_max_sync(FULL, on[j] && bin < 255 ? bin : 0);
        const int d = top - bin;
        const bool in = on[j] && d >= 0 && d < WIN;
#pragma unroll
        for (int i = 0; i < WIN; ++i) acc[i] += in && d == i ? val : 0;
        if (on[j] && !in) atomicAdd(bins + bin, (unsigned long long)val);
      }
    }
#pragma unroll
    for (int i = 0; i < WIN; ++i) {
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) acc[i] += __shfl_xor_sync(FULL, acc[i], d);
      if (lane == 0 && acc[i]) atomicAdd(bins + (top - i), (unsigned long long)acc[i]);
    }
  };
  for (uint32_t i = 0; i < P.cap; i += 1u << P.s) for_pieces(A, P.page(i), piece);
}

// The forest's edges into the warp's list, the state of its vertices as at the
// start; returns the entries.
__device__ __noinline__ unsigned list_forest(const Args &A, const Pages P, const Pages Q) {
  const int lane = threadIdx.x & 31;
  for (uint32_t i = lane; i < Q.cap; i += 32) {
    const int64_t v = Q.at(i);
    if (v >= A.n) continue;
    st_rel(A.p + v, (int32_t)v);
    A.r[v] = KEY_INF;
    A.roots[v] = (int32_t)v;
  }
  // a word of the bitmap per lane, whose bits it takes one after the other: all
  // lanes' gathers are in flight (edge by edge, R-MAT 20: 86 of the call's
  // 646 us; so the call takes 593)
  unsigned out = 0;
  for (uint32_t i0 = 0; i0 < P.cap; i0 += 1024) {
    const uint32_t i = i0 + 32 * lane;
    const int64_t e0 = P.at(i);
    uint32_t word = i < P.cap && e0 < A.m ? __ldcg(A.mbits + (e0 >> 5)) : 0u;
    const unsigned mine = (unsigned)__popc(word);
    unsigned incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned o = __shfl_up_sync(FULL, incl, d);
      if (lane >= d) incl += o;
    }
    unsigned at = out + incl - mine;
    out += __shfl_sync(FULL, incl, 31);
    for (; word; word &= word - 1u) {
      const int64_t e = e0 + __ffs((int)word) - 1;
      const int2 uv = A.ends[e];
      A.list[P.at(at++)] = make_uint4((uint32_t)uv.x, (uint32_t)uv.y, (uint32_t)e, ord_weight_dev(A.w[e], A.wtype));
    }
  }
  __syncwarp();
  return out;
}

// The rounds on the light classes (phase 0; the bitmap of the giant component
// when a heavy class follows) or on the heavy edges left (phase 1); the
// results at the end.  Phase 2 counts the rounds that the loop takes without
// classes: they are those on the forest's own edges (the lightest edge that
// leaves a component is one of them, so every round hooks the same roots).
template <bool BATCH, bool COUNT>
__global__ void __launch_bounds__(ET, 1) k_rounds(const __grid_constant__ Args A, int phase) {
  __shared__ BlockSums sums;
  __shared__ long long sbins[256];
  __shared__ Table tab;
  __shared__ unsigned s_live, s_pairs, s_edges;
  Ctrl *C = A.ctl;
  if (C->abort) return;  // (phase 0 did not finish)
  if (C->err) {          // an invalid edge: its indices must not be used
    if (blockIdx.x == 0 && threadIdx.x == 0) A.host[0] = C->err;
    return;
  }
  __shared__ GridBarrier bar;
  const int64_t tid = (int64_t)blockIdx.x * ET + threadIdx.x, nthr = (int64_t)gridDim.x * ET;
  const int64_t warp = tid >> 5;
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  unsigned long long usum = 0;  // uint32 weights of the thread's forest edges
  sums.clear();
  if (threadIdx.x == 0) {
    s_live = s_pairs = s_edges = 0;
    bar.init(C->arrive[phase], &C->abort);
  }
  table_clear(tab);
  __syncthreads();
  // the warp's vertices and its list of roots (all of them, or what the
  // flattening before the filter left)
  const Pages P(A.m, A.es, warp, nthr >> 5), Q(A.n, A.vs, warp, nthr >> 5);
  unsigned vc = phase == 1 ? A.back[warp] : Q.len;
  // the rounds are counted: those of phase 2, or of the only class
  const bool counting = COUNT && (phase == 2 || A.classes == 1);
  unsigned *pair_slot = C->pairs;
  int hooked = 0;       // rounds with hooks
  unsigned passes = 0;  // settling passes and chases
  auto counted = [&]() {  // (behind a grid barrier)
    if (!counting || tid != 0) return;
    A.host[1] = (unsigned)hooked;
    A.host[2] = hooked ? *(volatile unsigned *)&C->pairs[(hooked - 1) & 3] : 0u;
    A.host[3] = *(volatile unsigned *)&C->edges;
    A.host[4] = passes;
  };
  auto aborted = [&]() { return *(volatile unsigned *)&C->abort != 0; };
  // The block's table goes to r; then the grid meets and the warps' counts are
  // summed (0 when the wait ran out).
  auto total_live = [&](unsigned cnt) -> unsigned long long {
    if (lane == 0 && cnt) atomicAdd(&s_live, cnt);
    __syncthreads();
    for (int i = threadIdx.x; i < TS; i += ET) {
      const int32_t k = tab.key[i];
      const unsigned long long v = tab.val[i];
      if (k >= 0 && v < ld_rel64(A.r + k)) atomicMin(A.r + k, v);
    }
    table_clear(tab);  // (the thread's own slots)
    unsigned mine = 0;
    if (threadIdx.x == 0) {
      mine = s_live;
      s_live = 0;
      if (COUNT) {
        if (s_pairs) atomicAdd(pair_slot, s_pairs);
        if (s_edges) atomicAdd(&C->edges, s_edges);
        s_pairs = s_edges = 0;
      }
    }
    return bar.meet(mine) ? bar.sum : 0ull;
  };
  // The roots that hooked point to their new roots (Algorithm 3's chase of
  // the changed roots): passes of up to HOPS hops, each parent written by its
  // own thread only, until no chain is longer.  The list keeps the roots that
  // did not hook; a root without a minimum has no edge left and leaves it.
  // The minima are cleared on the way.
  auto settle_roots = [&]() -> bool {
    constexpr int U = 4;
    for (int pass = 0; pass < ROUND_CAP; ++pass) {
      ++passes;
      unsigned out = 0;
      bool more = false;
      for (unsigned b0 = 0; b0 < vc; b0 += 32 * U) {
        uint32_t k[U];
        int32_t x[U];
        unsigned long long rv[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
          const unsigned i = b0 + j * 32 + lane;
          k[j] = i < vc ? (uint32_t)A.roots[Q.at(i)] : 0xffffffffu;
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
          const bool on = k[j] != 0xffffffffu;
          const int32_t v = (int32_t)(k[j] & ~LONG);
          rv[j] = on && pass == 0 ? ld_rel64(A.r + v) : 0ull;
          x[j] = on && (pass == 0 || (k[j] & LONG)) ? ld_rel(A.p + v) : v;
        }
        int32_t y[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
          const int32_t v = (int32_t)(k[j] & ~LONG);
          y[j] = k[j] != 0xffffffffu && rv[j] != KEY_INF && x[j] != v ? __ldca(A.p + x[j]) : x[j];
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
          bool keep = k[j] != 0xffffffffu;
          const int32_t v = (int32_t)(k[j] & ~LONG);
          if (keep && rv[j] == KEY_INF) keep = false;
          if (keep && pass == 0) A.r[v] = KEY_INF;
          if (keep && x[j] != v) {
            int32_t a = x[j], b = y[j];
#pragma unroll 1
            for (int h = 0; h < HOPS && b != a; ++h) {
              a = b;
              b = __ldca(A.p + a);
            }
            if (a != x[j]) st_rel(A.p + v, a);
            keep = b != a;
            more |= keep;
            k[j] = (uint32_t)v | LONG;
          }
          const unsigned bal = __ballot_sync(FULL, keep);
          if (keep) A.roots[Q.at(out + __popc(bal & below))] = (int32_t)k[j];
          out += __popc(bal);
        }
      }
      __syncwarp();
      vc = out;
      const unsigned long long left = total_live(__any_sync(FULL, more) ? 1u : 0u);
      if (aborted()) return false;
      if (!left) return true;
    }
    return true;  // (a pass shortens every chain HOPS-fold: never reached)
  };
  // Every vertex points to its root (a chain has one hop per round at most),
  // the warp's list takes the roots among its vertices and, when asked for,
  // the bitmap the members of the tree `giant`.
  auto flatten = [&](bool bits, int32_t giant) -> bool {
    constexpr int U = 4;
    unsigned out = 0;
    int gv = 0;
    for (uint32_t i = 0; i < Q.cap; i += 32 * U) {
      const int64_t v0 = Q.at(i), vhi = A.n;
      if (BATCH && bits && !(i & ((1u << Q.s) - 1u))) gv = A.vg[Q.page(i)];
      int32_t x[U], y[U];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const int64_t v = v0 + j * 32 + lane;
        x[j] = v < vhi ? ld_rel(A.p + v) : -1;
      }
#pragma unroll
      for (int j = 0; j < U; ++j) y[j] = x[j] >= 0 ? __ldca(A.p + x[j]) : -1;
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const int64_t v = v0 + j * 32 + lane;
        int32_t a = x[j], b = y[j];
        while (b != a) {
          a = b;
          b = __ldca(A.p + a);
        }
        if (a != x[j]) st_rel(A.p + v, a);
        const bool root = v < vhi && a == (int32_t)v;
        const unsigned mr = __ballot_sync(FULL, root);
        if (root) A.roots[Q.at(out + __popc(mr & below))] = a;
        out += __popc(mr);
        if (bits) {
          if (BATCH && v < vhi) {
            gv = graph_from(A, gv, v);
            giant = A.giant[gv];
          }
          const unsigned mg = __ballot_sync(FULL, v < vhi && a == giant);
          if (lane == 0 && v < vhi) A.gbits[v >> 5] = mg;
        }
      }
    }
    __syncwarp();
    vc = out;
    return bar.meet();
  };
  // Rounds on the warp's `cnt` entries until no edge is left; the minima of
  // the first one have been offered.  With few edges left the roots are not
  // settled in a step of their own (a barrier and a pass over the roots, about
  // 5 us): the minimum pass follows the chains, all at the same time.
  auto rounds = [&](unsigned cnt) -> bool {
    unsigned long long live = total_live(cnt);
    for (int k = 0; k < ROUND_CAP && live; ++k) {
      const bool small = live <= (A.m > A.n + A.n / 4 ? SMALL : SMALL_CHAINS);
      const bool found = COUNT && phase == 2;  // (marked and summed before)
      const unsigned h = hook_pass(A, P, cnt, small, A.mbits && !found, !BATCH && A.totals && !found, sums, usum);
      if (counting) {  // (added up with the edges left; the round's slot was cleared two rounds before)
        const unsigned t = __reduce_add_sync(FULL, h & 0xffffu), q = __reduce_add_sync(FULL, h >> 16);
        if (lane == 0 && q) atomicAdd(&s_pairs, q);
        if (lane == 0 && t) atomicAdd(&s_edges, t);
        pair_slot = &C->pairs[k & 3];
        if (tid == 0) C->pairs[(k + 2) & 3] = 0;
        ++hooked;
      }
      if (!bar.meet()) return false;
      if (!small) {
        if (!settle_roots()) return false;
        cnt = min_pass<true, false>(A, tab, P, 0u, cnt);
      } else {
        ++passes;
        cnt = min_pass<true, true>(A, tab, P, 0u, cnt);
      }
      live = total_live(cnt);
    }
    return !aborted();
  };

  unsigned cnt;
  if (COUNT && phase == 2) {
    cnt = list_forest(A, P, Q);
    if (!bar.meet()) return;
  } else {
    cnt = A.front[warp];
  }
  cnt = min_pass<false, false>(A, tab, P, 0u, cnt);
  if (!rounds(cnt)) return;
  if (COUNT && phase == 2) {
    counted();
    return;
  }
  if (phase == 0 && A.second) {
    if (!flatten(false, 0)) return;
    const unsigned back = A.back[warp];
    cnt = min_pass<true, false>(A, tab, P, P.cap - back, back);
    if (!rounds(cnt)) return;
  }
  const bool last = phase == 1 || A.classes < 3;
  if (!last) {
    if (BATCH) {
      vote_giants(A, warp, nthr >> 5);
      if (!bar.meet()) return;
    }
    flatten(true, BATCH ? 0 : vote_giant(A));
    if (lane == 0) A.back[warp] = vc;
  }
  // the forest's weight so far (a batch: from the bitmap, at the end)
  if (!BATCH && A.totals) {
    if (A.wtype == MSF_U32) {
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) usum += __shfl_xor_sync(FULL, usum, d);
      if (lane == 0 && usum) atomicAdd(A.bins, usum);
    } else {
      __syncthreads();
      for (int i = threadIdx.x; i < 256; i += ET) {
        const unsigned long long v = sums.get(i);
        if (v) atomicAdd(A.bins + i, v);
      }
    }
  }
  if (!last) return;
  // results.  The smallest vertex of every tree: r is all KEY_INF again, and
  // the low half of a root's word takes the minimum of the tree's other
  // vertices (through the block's table); a label is the smaller of it and the
  // root.
  constexpr int U = 4;
  if (A.labels) {
    for (uint32_t i = 0; i < Q.cap; i += 32 * U) {
      const int64_t v0 = Q.at(i), vhi = A.n;
      int32_t x[U], y[U];
#pragma unroll
      for (int j = 0; j < U; ++j) x[j] = v0 + j * 32 + lane < vhi ? ld_rel(A.p + v0 + j * 32 + lane) : 0;
#pragma unroll
      for (int j = 0; j < U; ++j) y[j] = __ldca(A.p + x[j]);
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const int64_t v = v0 + j * 32 + lane;
        if (v >= vhi) continue;
        int32_t a = x[j], b = y[j];
        while (b != a) {
          a = b;
          b = __ldca(A.p + a);
        }
        if (a != x[j]) st_rel(A.p + v, a);
        if (a <= (int32_t)v) continue;  // (the root itself is added when read)
        bool hit;
        const int slot = table_slot(tab, a, hit);
        unsigned *low = reinterpret_cast<unsigned *>(slot < 0 ? A.r + a : tab.val + slot);
        if (slot < 0 || (unsigned)v < *(volatile unsigned *)low) atomicMin(low, (unsigned)v);
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < TS; i += ET) {
      const unsigned b = *reinterpret_cast<unsigned *>(tab.val + i);
      if (tab.key[i] >= 0 && b != 0xffffffffu) atomicMin(reinterpret_cast<unsigned *>(A.r + tab.key[i]), b);
    }
  }
  if (!bar.meet()) return;
  if (!BATCH && A.totals && blockIdx.x == 0) {
    for (int i = threadIdx.x; i < 256; i += ET) sbins[i] = (long long)ld_rel64(A.bins + i);
    __syncthreads();
    if (threadIdx.x < 32) {
      const double t = combine_bins_warp(sbins, A.wtype);
      if (threadIdx.x == 0) *A.totals = t;
    }
  }
  if (A.labels) {
    int gv = 0;
    for (uint32_t i = 0; i < Q.cap; i += 32 * U) {
      const int64_t v0 = Q.at(i), vhi = A.n;
      if (BATCH && !(i & ((1u << Q.s) - 1u))) gv = A.vg[Q.page(i)];
      int32_t x[U];
      unsigned b[U];
#pragma unroll
      for (int j = 0; j < U; ++j) x[j] = v0 + j * 32 + lane < vhi ? __ldca(A.p + v0 + j * 32 + lane) : 0;
#pragma unroll
      for (int j = 0; j < U; ++j) b[j] = __ldca(reinterpret_cast<const unsigned *>(A.r + x[j]));
#pragma unroll
      for (int j = 0; j < U; ++j)
        if (v0 + j * 32 + lane < vhi) {
          const int64_t v = v0 + j * 32 + lane;
          const int32_t least = (int32_t)min(b[j], (unsigned)x[j]);
          if (BATCH) {
            gv = graph_from(A, gv, v);
            A.labels[A.vA[gv] + (v - A.vL[gv])] = least - (int32_t)A.vL[gv];
          } else {
            A.labels[v] = least;
          }
        }
    }
  }
  if (BATCH) {
    batch_results(A, P);
    if (A.totals) {
      if (!bar.meet()) return;
      // a warp per graph rounds its total
      for (int64_t g = warp; g < A.G; g += nthr >> 5) {
        const double t = combine_bins_warp(reinterpret_cast<const long long *>(A.bins) + g * 256, A.wtype);
        if (lane == 0) A.totals[A.id[g]] = t;
      }
    }
    if (tid == 0) A.host[0] = *(volatile unsigned *)&C->err;
    return;
  }
  if (A.mask) {
    const int64_t m = A.m;
    const int64_t head = (int64_t)((16 - (reinterpret_cast<uintptr_t>(A.mask) & 15)) & 15);
    const int64_t h = head < m ? head : m;
    const int64_t nq = (m - h) >> 4;
    uint4 *q = reinterpret_cast<uint4 *>(A.mask + h);
    for (int64_t e = tid; e < h; e += nthr) A.mask[e] = (uint8_t)((A.mbits[e >> 5] >> (e & 31)) & 1u);
    for (int64_t i = tid; i < nq; i += nthr) q[i] = spread16(bits16(A.mbits, h + (i << 4)));
    for (int64_t e = h + (nq << 4) + tid; e < m; e += nthr)
      A.mask[e] = (uint8_t)((A.mbits[e >> 5] >> (e & 31)) & 1u);
  }
  counted();
  if (tid == 0) A.host[0] = *(volatile unsigned *)&C->err;
}

size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

// The edges as separate arrays (src, dst) or as pairs of validated ends; with
// `counts` (one graph, pairs) the rounds of the loop without classes too.
int solve(int32_t K, const int32_t *which, const int64_t *voff, const int64_t *eoff, const int32_t *src,
          const int32_t *dst, const int2 *ends, const uint32_t *w, int wtype, uint8_t *mask, int32_t *labels,
          double *totals, unsigned *status, LoopCounts *counts, int32_t spare, cudaStream_t s) {
  int64_t n = 0, m = 0;
  if (!which) {
    n = voff[1];
    m = eoff[1];
  }
  for (int32_t k = 0; which && k < K; ++k) {
    n += voff[which[k] + 1] - voff[which[k]];
    m += eoff[which[k] + 1] - eoff[which[k]];
  }
  Args A;
  std::memset(&A, 0, sizeof(A));
  A.n = n;
  A.m = m;
  A.src = src;
  A.dst = dst;
  A.ends = ends;
  A.w = w;
  A.wtype = wtype;
  const bool vec = ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst) |
                     reinterpret_cast<uintptr_t>(w)) & 15) == 0;
  // blocks: one per BLOCK_SHARE edges or vertices, at most one per SM
  int64_t want = ((m > n ? m : n) + BLOCK_SHARE - 1) / BLOCK_SHARE;
  if (want < 1) want = 1;
  DeviceShare share(n, m);
  int64_t cap = (int64_t)sm_count() - spare;  // (other blocks run on `spare` SMs meanwhile)
  if (cap > share.sms) cap = share.sms;
  const int blocks = (int)(want < cap ? want : cap);
  const int64_t warps = (int64_t)blocks * EW;
  A.es = page_shift(m, warps);
  A.vs = page_shift(n, warps);
  const int64_t epages = page_count(m, A.es), vpages = page_count(n, A.vs);
  A.classes = 1;
  if (m >= 64 * SAMPLES && (!counts || count_by_replay(n, m))) {
    double la = CLASS1, lb = CLASS2;
    if (!two_classes(n, m)) la = lb;
    if ((double)m > 1.25 * la * (double)n && la < lb) A.classes = 2;
    if ((double)m > 1.25 * lb * (double)n) A.classes = 3;
    A.second = A.classes > 1 && la < lb;
    A.rank[0] = (unsigned)light_rank(la, n, m, SAMPLES, la < lb ? 8 : 16);
    A.rank[1] = (unsigned)light_rank(lb, n, m, SAMPLES, 16);
  }
  const size_t bit_bytes = (size_t)((n + 127) / 128) * 16;
  A.smem_bits = A.classes > 2 && bit_bytes <= SMEM_BITS;
  const size_t dyn = A.smem_bits ? bit_bytes : 0;
  size_t off = 0;
  auto place = [&](size_t bytes) {
    const size_t at = off;
    off = align_up(off + bytes);
    return at;
  };
  static_assert(sizeof(Ctrl) <= 256, "control block");
  const size_t ctl_bytes = 256 + 256 * 8;  // control block, long accumulators
  const size_t tab_bytes = which ? (size_t)(K + 1) * 32 + (size_t)K * 4 : 0;  // eL, vL, eA, vA, id
  const size_t o_tab = place(tab_bytes), o_giant = place((size_t)(which ? K : 0) * 4);
  const size_t o_bbins = place((size_t)(which ? K : 0) * 256 * 8);
  const size_t o_ctl = place(ctl_bytes), o_p = place((size_t)(n + 1) * 4), o_r = place((size_t)(n + 1) * 8);
  const size_t o_roots = place(((size_t)vpages << A.vs) * 4), o_gbits = place(bit_bytes);
  const size_t o_bits = place(((size_t)(m + 31) / 32 + 2) * 4);
  const size_t o_front = place((size_t)warps * 4), o_back = place((size_t)warps * 4);
  const size_t o_eg = place(which ? (size_t)epages * 4 : 0), o_vg = place(which ? (size_t)vpages * 4 : 0);
  const size_t o_list = place(((size_t)epages << A.es) * 16);
  int err = MSF_OK;
  char *base = (char *)pool_alloc(off, &err);
  if (err) return err;
  PoolBlock back{base};
  PinnedWords pin;
  if (int rc = pin.take(64 + tab_bytes)) return rc;
  Settle settle(s);
  pin.p[0] = 0x80000000u;  // not finished
  pin.p[1] = counts ? 0x80000000u : 0u;
  A.ctl = (Ctrl *)(base + o_ctl);
  A.p = (int32_t *)(base + o_p);
  A.r = (unsigned long long *)(base + o_r);
  A.roots = (int32_t *)(base + o_roots);
  A.gbits = (uint32_t *)(base + o_gbits);
  // the mask comes from the bitmap, and so do a batch's totals and the replay's list
  A.mbits = mask || (which && totals) || (counts && A.classes > 1) ? (uint32_t *)(base + o_bits) : nullptr;
  A.bins = (unsigned long long *)(base + o_ctl + 256);
  A.front = (unsigned *)(base + o_front);
  A.back = (unsigned *)(base + o_back);
  A.list = (uint4 *)(base + o_list);
  A.mask = mask;
  A.labels = labels;
  A.totals = totals;
  A.host = pin.p;
  if (which) {
    int64_t *t = (int64_t *)(pin.p + 16);
    int32_t *ids = (int32_t *)(t + 4 * (K + 1));
    int64_t *eL = t, *vL = t + (K + 1), *eA = t + 2 * (K + 1), *vA = t + 3 * (K + 1);
    eL[0] = vL[0] = 0;
    for (int32_t k = 0; k < K; ++k) {
      const int32_t g = which[k];
      eL[k + 1] = eL[k] + (eoff[g + 1] - eoff[g]);
      vL[k + 1] = vL[k] + (voff[g + 1] - voff[g]);
      eA[k] = eoff[g];
      vA[k] = voff[g];
      ids[k] = g;
    }
    eA[K] = vA[K] = 0;
    int64_t *d = (int64_t *)(base + o_tab);
    MSF_CK(cudaMemcpyAsync(d, t, tab_bytes, cudaMemcpyHostToDevice, s));
    A.G = K;
    A.eL = d;
    A.vL = d + (K + 1);
    A.eA = d + 2 * (K + 1);
    A.vA = d + 3 * (K + 1);
    A.id = (int32_t *)(d + 4 * (K + 1));
    A.giant = (int32_t *)(base + o_giant);
    A.eg = (int32_t *)(base + o_eg);
    A.vg = (int32_t *)(base + o_vg);
    A.bins = (unsigned long long *)(base + o_bbins);
  }
  MSF_CK(cudaMemsetAsync(A.ctl, 0, ctl_bytes, s));
  k_prepare<<<blocks, ET, 0, s>>>(A);
  const bool f32 = wtype == MSF_F32;
  void (*select)(Args) =
      which  ? (f32 ? (vec ? k_select<VECTOR, true, true> : k_select<SCALAR, true, true>)
                    : (vec ? k_select<VECTOR, false, true> : k_select<SCALAR, false, true>))
      : ends ? (f32 ? k_select<PAIRS, true, false> : k_select<PAIRS, false, false>)
             : (f32 ? (vec ? k_select<VECTOR, true, false> : k_select<SCALAR, true, false>)
                    : (vec ? k_select<VECTOR, false, false> : k_select<SCALAR, false, false>));
  const void *rounds = which    ? (const void *)k_rounds<true, false>
                       : counts ? (const void *)k_rounds<false, true>
                                : (const void *)k_rounds<false, false>;
  select<<<blocks, ET, 0, s>>>(A);
  int phase = 0;
  void *args[] = {&A, &phase};
  cudaError_t e = cudaLaunchCooperativeKernel(rounds, dim3((unsigned)blocks), dim3(ET), args, 0, s);
  if (e == cudaSuccess && A.classes > 2) {
    void (*filter)(Args) =
        which  ? (A.smem_bits ? (vec ? k_filter<VECTOR, true, true> : k_filter<SCALAR, true, true>)
                              : (vec ? k_filter<VECTOR, false, true> : k_filter<SCALAR, false, true>))
        : ends ? (A.smem_bits ? k_filter<PAIRS, true, false> : k_filter<PAIRS, false, false>)
               : (A.smem_bits ? (vec ? k_filter<VECTOR, true, false> : k_filter<SCALAR, true, false>)
                              : (vec ? k_filter<VECTOR, false, false> : k_filter<SCALAR, false, false>));
    if (A.smem_bits)
      e = cudaFuncSetAttribute(filter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BITS);
    if (e == cudaSuccess) {
      filter<<<blocks, ET, dyn, s>>>(A);
      phase = 1;
      e = cudaLaunchCooperativeKernel(rounds, dim3((unsigned)blocks), dim3(ET), args, 0, s);
    }
  }
  if (e == cudaSuccess && counts && A.classes > 1) {
    phase = 2;
    e = cudaLaunchCooperativeKernel(rounds, dim3((unsigned)blocks), dim3(ET), args, 0, s);
  }
  if (e == cudaErrorCooperativeLaunchTooLarge) {  // (a share of the device that holds fewer blocks)
    cudaGetLastError();
    MSF_CK(cudaStreamSynchronize(s));
    return SOLVE_NOT_RUN;
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  const cudaError_t e2 = cudaStreamSynchronize(s);
  settle.done = true;
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) return cuda_fail(e, "forest of an edge list");
  const unsigned st = *(volatile unsigned *)pin.p;
  if ((st | pin.p[1]) & 0x80000000u) return fail(MSF_ERR_CHECK, "device consistency check failed");
  *status |= st;
  if (counts) {
    counts->hooked = (int32_t)pin.p[1];
    counts->left = pin.p[2];
    counts->edges = pin.p[3];
    counts->passes = (int32_t)pin.p[4];
    counts->kernels = 3 + (A.classes > 2 ? 2 : 0) + (A.classes > 1 ? 1 : 0);
  }
  return MSF_OK;
}

}  // namespace

// Forest of one graph from its edge list, or of K graphs of a batch, `which` of
// the graphs with the host offsets voff, eoff (pointers the device can read).
// Any output may be NULL.  Synchronizes `s`; *status: 1 = index out of range,
// 2 = NaN weight.
int solve_edges(int32_t K, const int32_t *which, const int64_t *voff, const int64_t *eoff, const int32_t *src,
                const int32_t *dst, const uint32_t *w, int wtype, uint8_t *mask, int32_t *labels, double *totals,
                unsigned *status, int32_t spare, cudaStream_t s) {
  return solve(K, which, voff, eoff, src, dst, nullptr, w, wtype, mask, labels, totals, status, nullptr, spare, s);
}

int solve_pairs(int64_t n, int64_t m, const int2 *ends, const uint32_t *w, int wtype, uint8_t *mask, int32_t *labels,
                double *totals, LoopCounts *counts, cudaStream_t s) {
  const int64_t voff[2] = {0, n}, eoff[2] = {0, m};
  unsigned status = 0;
  return solve(1, nullptr, voff, eoff, nullptr, nullptr, ends, w, wtype, mask, labels, totals, &status, counts, 0, s);
}

}  // namespace msf
