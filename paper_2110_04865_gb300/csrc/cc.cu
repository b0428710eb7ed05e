// Connected components (Sec. 2.4) from the edges the build kept, in one
// cooperative kernel.
//
// The rounds are those of the loop over the CSR, step for step (the round count
// is a statistic, so no other method will do): conditional hooking, starcheck,
// unconditional hooking, complete shortcutting.  The loop sweeps every slot of
// the CSR twice a round, about 240 us each for 2^24 edges.  Here an edge offers
// to both ends at once, and most edges are read without a gathered parent:
//
//   first conditional       parents are the vertices themselves: an edge offers
//                           its smaller end to its larger one;
//   first unconditional     only an edge between a star and another tree has
//                           something to offer: two bits of the star bitmap
//                           tell, from shared memory when it fits there;
//   second conditional      an edge inside the giant tree has nothing to offer
//                           any more: two bits of its bitmap tell.  The edges
//                           between trees go to the warps' lists, and all later
//                           steps read and compact those.
//
// R-MAT 20 with 2^24 edges, us: the first pass 91 (one gather an edge), the two
// that read bitmaps 69 (instruction issue) and 145 (the parents of the edges
// between trees, and their list), the lists 43 and 31, the passes over the
// vertices 3 to 10 each, barriers 1 to 2 each.  The call (loop over the CSR
// before, this after): R-MAT 20 1466 -> 466 us, uniform 2^24 edges 1429 -> 520,
// 96^3 lattice 278 -> 98, R-MAT 16 157 -> 86, 1296 vertices 142 -> 39.
// Variants that measured slower: a block's recent offers kept in a table (first
// pass 104, second bitmap pass 199), byte flags for the starcheck (72 against 9).
#include <cstring>

#include "exact.cuh"
#include "grid.cuh"
#include "internal.cuh"

namespace msf {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int CT = 1024;        // threads per block, one block per SM
constexpr int CW = CT / 32;     // warps per block
constexpr int VOTES = 128;      // sampled edge ends for the giant tree
constexpr int HOPS = 16;        // hops of one settling pass
constexpr int ROUND_CAP = 64;
constexpr size_t CC_BITS = 224 << 10;  // largest bitmap kept in shared memory
// Entries of the lists from which a round's first step reads the giant tree's
// bitmap before the parents (its making costs about 7 us at 2^20 vertices).
constexpr unsigned LONG_LIST = 1u << 12;  // (in units of 256)
constexpr uint32_t NONE = 0xffffffffu;
// Up to FEW vertices of many edges each the first offers are collected per block.
// Calls in us at (vertices, edges), loop over the CSR / edge by edge / collected:
// (30, 10^6) 150 / 175 / 62, (300, 500 000) 131 / 161 / 63, (300, 2 M) 163 / 191 / 66,
// (2000, 500 000) 192 / 117 / 88; (2000, 60 000) 182 / 81 / 84, (1296, 5000) 180 / 62
// / 70.
constexpr int64_t FEW = 2048;
// Edges or vertices per block of a call that does not fill the device; one block
// up to ONE_BLOCK of them, whose barriers are its own (whole calls in us, several
// blocks / one, uniform: 2000 edges 60 / 45, 5000 65 / 55, 10 000 65 / 61).
constexpr int64_t BLOCK_SHARE = 4096, ONE_BLOCK = 8192;

struct CcCtrl {
  unsigned long long arrive[2];
  unsigned abort;
};

struct CcArgs {
  int64_t n, m;
  const int2 *ends;
  int32_t es, vs;      // pages of 2^es edges and 2^vs vertices
  int32_t smem_bits;   // a bitmap of the vertices fits in shared memory
  int32_t few;         // the first offers are collected per block
  int32_t *p;          // parents
  uint32_t *q;         // smallest offered parent of each root
  uint32_t *deep;      // bitmap: roots of trees that are not stars (and some of their vertices)
  uint32_t *bits;      // star vertices, then the giant tree's
  int2 *list;          // edges between trees, a region per warp
  CcCtrl *ctl;
  int32_t *labels;
  unsigned *host;      // pinned: [0] not finished, [1] rounds
};

// Four edges of a lane.
struct PairQuad {
  int4 s, d;
};

// Lowers a root's offer.  A q read out of date is never too small.  Until q is
// lowered everything in flight passes the test (600 000 threads' edges, each about
// 1 ns on one word): lanes with the first one's root send their smallest offer.
__device__ __forceinline__ void lower(uint32_t *q, int32_t root, uint32_t parent) {
  const unsigned m = __activemask();
  const int first = __ffs((int)m) - 1;
  const unsigned same = __ballot_sync(m, root == __shfl_sync(m, root, first));
  if (!(same >> (threadIdx.x & 31) & 1u)) {
    atomicMin(q + root, parent);
    return;
  }
  const unsigned least = __reduce_min_sync(same, parent);
  if ((int)(threadIdx.x & 31) == first) atomicMin(q + root, least);
}
__device__ __forceinline__ void offer(uint32_t *q, int32_t root, int32_t parent) {
  if ((uint32_t)parent < __ldca(q + root)) lower(q, root, (uint32_t)parent);
}

__global__ void __launch_bounds__(CT, 1) k_components(const __grid_constant__ CcArgs A) {
  extern __shared__ uint32_t dyn[];
  __shared__ unsigned s_list;
  __shared__ int32_t vote[VOTES];
  __shared__ unsigned best;
  CcCtrl *C = A.ctl;
  const int64_t tid = (int64_t)blockIdx.x * CT + threadIdx.x, warps = (int64_t)gridDim.x * CW;
  const int64_t warp = tid >> 5;
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  const Pages P(A.m, A.es, warp, warps), Q(A.n, A.vs, warp, warps);
  const int64_t n = A.n, m = A.m;
  int32_t *p = A.p;
  uint32_t *q = A.q;
  __shared__ GridBarrier bar;
  constexpr int U = 4;
  auto barrier = [&]() { return bar.meet(); };
  // Barrier; whether a thread of the grid has `some`, and the length of all lists
  // in units of 256 entries a block.
  unsigned cnt = 0;   // entries of the warp's list
  unsigned live = 0;  // of all, in those units
  int32_t giant = -1;
  auto total = [&](bool some, bool &any) -> bool {
    if (lane == 0 && cnt) atomicAdd(&s_list, cnt);
    some = __syncthreads_or(some);
    unsigned long long mine = 0;
    if (threadIdx.x == 0) {
      mine = ((unsigned long long)(some ? 1u : 0u) << 36) + (s_list >> 8);
      s_list = 0;
    }
    if (!bar.meet(mine)) return false;
    any = bar.sum >> 36 != 0;
    live = (unsigned)(bar.sum & ((1ull << 36) - 1ull));
    return true;
  };
  // The warp's vertices in groups of U * 32 (a group lies in one page).
  auto vertices = [&](auto f) {
    for (uint32_t i = 0; i < Q.cap; i += 32 * U) f(Q.at(i));
  };
  // Roots with an offer take it; whether one of the thread's did.
  auto hook = [&]() -> bool {
    bool c = false;
    vertices([&](int64_t v0) {
      uint32_t x[U];
#pragma unroll
      for (int j = 0; j < U; ++j) x[j] = v0 + j * 32 + lane < n ? __ldcg(q + v0 + j * 32 + lane) : NONE;
#pragma unroll
      for (int j = 0; j < U; ++j) {
        if (x[j] == NONE) continue;
        const int64_t v = v0 + j * 32 + lane;
        q[v] = NONE;
        p[v] = (int32_t)x[j];
        c = true;
      }
    });
    return c;
  };
  // The bitmap where the passes over all edges read it.
  auto bitmap = [&]() -> const uint32_t * {
    if (!A.smem_bits) return A.bits;
    const int64_t words = (n + 31) / 32;
    for (int64_t i = threadIdx.x; i < words; i += CT) dyn[i] = __ldcg(A.bits + i);
    __syncthreads();
    return dyn;
  };
  auto load = [&](int b) {
    PairQuad x;
    x.s = x.d = make_int4(0, 0, 0, 0);  // (zeros past the end: self-loops)
    load_pairs(A.ends, P.at((uint32_t)b) + 4 * lane, (uint32_t)b < P.cap ? m : 0, x.s, x.d);
    return x;
  };
  // Roots of the list's edges, those inside a tree dropped; the others offer.
  auto conditional_list = [&]() -> unsigned {
    const uint32_t *bits = live > LONG_LIST ? bitmap() : nullptr;
    unsigned out = 0;
    for (unsigned b0 = 0; b0 < cnt; b0 += 32 * U) {
      int2 x[U];
      int32_t a[U], b[U];
      bool any = false;
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const unsigned i = b0 + j * 32 + lane;
        x[j] = i < cnt ? A.list[P.at(i)] : make_int2(0, 0);
      }
#pragma unroll
      for (int j = 0; j < U; ++j) {
        if (bits && (bits[(uint32_t)x[j].x >> 5] >> (x[j].x & 31)) & (bits[(uint32_t)x[j].y >> 5] >> (x[j].y & 31)) & 1u)
          x[j] = make_int2(0, 0);
        any |= x[j].x != x[j].y;
      }
      if (!__any_sync(FULL, any)) continue;
#pragma unroll
      for (int j = 0; j < U; ++j) {
        a[j] = __ldca(p + x[j].x);
        b[j] = __ldca(p + x[j].y);
      }
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const bool on = a[j] != b[j];
        const unsigned bal = __ballot_sync(FULL, on);
        if (on) {
          offer(q, max(a[j], b[j]), min(a[j], b[j]));
          A.list[P.at(out + __popc(bal & below))] = x[j];
        }
        out += __popc(bal);
      }
    }
    __syncwarp();
    return out;
  };

  if (threadIdx.x == 0) {
    s_list = 0;
    bar.init(C->arrive, &C->abort);
  }
  vertices([&](int64_t v0) {
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int64_t v = v0 + j * 32 + lane;
      if (v >= n) continue;
      p[v] = (int32_t)v;
      q[v] = NONE;
      if (lane == 0) A.deep[v >> 5] = 0u;
    }
  });
  if (!barrier()) return;
  int round = 0;
  for (;; ++round) {
    if (round == ROUND_CAP) {
      if (tid == 0) A.host[0] = 2u;
      return;
    }
    // conditional hooking: every tree is a star
    if (round == 0 && A.few) {
      // few vertices: their offers meet in the block first (an edge would find
      // q as it was when its line came to L1, and most edges would offer)
      for (int i = threadIdx.x; i < (int)n; i += CT) dyn[i] = NONE;
      __syncthreads();
      auto body = [&](const PairQuad &x, int) {
        const int32_t u[4] = {x.s.x, x.s.y, x.s.z, x.s.w}, v[4] = {x.d.x, x.d.y, x.d.z, x.d.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int32_t lo = min(u[j], v[j]), hi = max(u[j], v[j]);
          if (lo != hi && (uint32_t)lo < *(volatile uint32_t *)(dyn + hi)) atomicMin(dyn + hi, (uint32_t)lo);
        }
      };
      stream2<PairQuad>(0, (int)P.cap, load, body);
      __syncthreads();
      for (int i = threadIdx.x; i < (int)n; i += CT)
        if (dyn[i] != NONE) offer(q, i, (int32_t)dyn[i]);
    } else if (round == 0) {
      auto body = [&](const PairQuad &x, int) {
        const int32_t u[4] = {x.s.x, x.s.y, x.s.z, x.s.w}, v[4] = {x.d.x, x.d.y, x.d.z, x.d.w};
        uint32_t old[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) old[j] = __ldca(q + max(u[j], v[j]));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int32_t lo = min(u[j], v[j]), hi = max(u[j], v[j]);
          if (lo != hi && (uint32_t)lo < old[j]) lower(q, hi, (uint32_t)lo);
        }
      };
      stream2<PairQuad>(0, (int)P.cap, load, body);
    } else if (round == 1) {
      const uint32_t *bits = bitmap();
      auto body = [&](const PairQuad &x, int) {
        const int32_t u[4] = {x.s.x, x.s.y, x.s.z, x.s.w}, v[4] = {x.d.x, x.d.y, x.d.z, x.d.w};
        unsigned iu[4], iv[4];  // (a giant's vertex needs no gathered parent)
        bool any = false;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          iu[j] = (bits[(uint32_t)u[j] >> 5] >> (u[j] & 31)) & 1u;
          iv[j] = (bits[(uint32_t)v[j] >> 5] >> (v[j] & 31)) & 1u;
          any |= !(iu[j] & iv[j]);
        }
        if (!__any_sync(FULL, any)) return;
        int32_t a[4], b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          a[j] = iu[j] ? giant : __ldca(p + u[j]);
          b[j] = iv[j] ? giant : __ldca(p + v[j]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const bool on = a[j] != b[j];
          const unsigned bal = __ballot_sync(FULL, on);
          if (on) {
            offer(q, max(a[j], b[j]), min(a[j], b[j]));
            A.list[P.at(cnt + __popc(bal & below))] = make_int2(u[j], v[j]);
          }
          cnt += __popc(bal);
        }
      };
      stream2<PairQuad>(0, (int)P.cap, load, body);
      __syncwarp();
    } else {
      cnt = conditional_list();
    }
    if (!barrier()) return;
    bool hooks;
    if (!total(hook(), hooks)) return;
    if (!hooks) break;  // (every tree is a star: the second step finds no other)
    // starcheck: a vertex whose parent is no root marks its grandparent; a tree
    // that is no star has a marked root.  Few vertices are marked by many, so a
    // block collects its marks first (bytes written at once: 72 us, R-MAT 20).
    uint32_t *marks = A.smem_bits ? dyn : A.deep;
    const int64_t words = (n + 31) / 32;
    if (A.smem_bits) {
      for (int64_t i = threadIdx.x; i < words; i += CT) dyn[i] = 0u;
      __syncthreads();
    }
    vertices([&](int64_t v0) {
      int32_t x[U], y[U];
#pragma unroll
      for (int j = 0; j < U; ++j) x[j] = v0 + j * 32 + lane < n ? __ldca(p + v0 + j * 32 + lane) : 0;
#pragma unroll
      for (int j = 0; j < U; ++j) y[j] = __ldca(p + x[j]);
#pragma unroll
      for (int j = 0; j < U; ++j) {
        if (v0 + j * 32 + lane >= n || x[j] == y[j]) continue;
        uint32_t *at = marks + (y[j] >> 5);
        if (!(*(volatile uint32_t *)at >> (y[j] & 31) & 1u)) atomicOr(at, 1u << (y[j] & 31));
      }
    });
    if (A.smem_bits) {
      __syncthreads();
      for (int64_t i = threadIdx.x; i < words; i += CT)
        if (dyn[i]) atomicOr(A.deep + i, dyn[i]);
    }
    if (!barrier()) return;
    vertices([&](int64_t v0) {
      int32_t x[U], y[U];
#pragma unroll
      for (int j = 0; j < U; ++j) x[j] = v0 + j * 32 + lane < n ? __ldca(p + v0 + j * 32 + lane) : 0;
#pragma unroll
      for (int j = 0; j < U; ++j) y[j] = __ldca(p + x[j]);
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const int64_t v = v0 + j * 32 + lane;
        const bool star = v < n && x[j] == y[j] && !(__ldca(A.deep + (x[j] >> 5)) >> (x[j] & 31) & 1u);
        const unsigned b = __ballot_sync(FULL, star);
        if (lane == 0 && v < n) A.bits[v >> 5] = b;
      }
    });
    if (!barrier()) return;
    // unconditional hooking: a star's vertex offers its root the parent of a
    // neighbour outside of stars
    if (round == 0) {
      const uint32_t *bits = bitmap();
      auto body = [&](const PairQuad &x, int) {
        const int32_t u[4] = {x.s.x, x.s.y, x.s.z, x.s.w}, v[4] = {x.d.x, x.d.y, x.d.z, x.d.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const unsigned su = (bits[(uint32_t)u[j] >> 5] >> (u[j] & 31)) & 1u;
          const unsigned sv = (bits[(uint32_t)v[j] >> 5] >> (v[j] & 31)) & 1u;
          if (su != sv) offer(q, __ldca(p + (su ? u[j] : v[j])), __ldca(p + (su ? v[j] : u[j])));
        }
      };
      stream2<PairQuad>(0, (int)P.cap, load, body);
    } else {
      const uint32_t *bits = bitmap();
      for (unsigned b0 = 0; b0 < cnt; b0 += 32 * U) {
        int2 x[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
          const unsigned i = b0 + j * 32 + lane;
          x[j] = i < cnt ? A.list[P.at(i)] : make_int2(0, 0);
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
          const unsigned su = (bits[(uint32_t)x[j].x >> 5] >> (x[j].x & 31)) & 1u;
          const unsigned sv = (bits[(uint32_t)x[j].y >> 5] >> (x[j].y & 31)) & 1u;
          if (su != sv) offer(q, __ldca(p + (su ? x[j].x : x[j].y)), __ldca(p + (su ? x[j].y : x[j].x)));
        }
      }
    }
    if (!barrier()) return;
    hook();
    if (!barrier()) return;
    // complete shortcutting: passes of up to HOPS hops, each parent written by
    // its own thread only (a parent read meanwhile is an ancestor)
    for (int pass = 0; pass < ROUND_CAP; ++pass) {
      bool more = false;
      vertices([&](int64_t v0) {
        int32_t x[U], y[U], a[U];
        bool any = false;
#pragma unroll
        for (int j = 0; j < U; ++j) x[j] = v0 + j * 32 + lane < n ? ld_rel(p + v0 + j * 32 + lane) : -1;
#pragma unroll
        for (int j = 0; j < U; ++j) y[j] = x[j] >= 0 ? __ldca(p + x[j]) : -1;  // (no vertex: no chain)
#pragma unroll
        for (int j = 0; j < U; ++j) {
          const int64_t v = v0 + j * 32 + lane;
          if (v < n && pass == 0 && lane == 0) A.deep[v >> 5] = 0u;
          a[j] = x[j];
          any |= a[j] != y[j];
        }
#pragma unroll 1
        for (int h = 0; h < HOPS && any; ++h) {  // (the lane's chains side by side)
          any = false;
#pragma unroll
          for (int j = 0; j < U; ++j) {
            const int32_t z = a[j] != y[j] ? __ldca(p + y[j]) : y[j];
            a[j] = y[j];
            y[j] = z;
            any |= a[j] != z;
          }
        }
        more |= any;
#pragma unroll
        for (int j = 0; j < U; ++j)
          if (a[j] != x[j]) st_rel(p + v0 + j * 32 + lane, a[j]);
      });
      bool left;
      if (!total(more, left)) return;
      if (!left) break;
    }
    if (round == 0 || live > LONG_LIST) {
      // the giant tree: the root that most of the sampled edge ends lie under
      // (every block finds the same one), as a bitmap
      if (threadIdx.x == 0) best = 0;
      if (threadIdx.x < VOTES) {
        int32_t x = 0;
        if (m > 0) {
          const int2 e = A.ends[(int64_t)((unsigned long long)threadIdx.x * (unsigned long long)m / VOTES)];
          x = (threadIdx.x & 1) ? e.x : e.y;
        }
        vote[threadIdx.x] = __ldca(p + x);
      }
      __syncthreads();
      if (threadIdx.x < VOTES) {
        unsigned c = 0;
        for (int i = 0; i < VOTES; ++i) c += vote[i] == vote[threadIdx.x];
        atomicMax(&best, (c << 16) | threadIdx.x);
      }
      __syncthreads();
      giant = vote[best & 0xffffu];
      vertices([&](int64_t v0) {
#pragma unroll
        for (int j = 0; j < U; ++j) {
          const int64_t v = v0 + j * 32 + lane;
          const unsigned b = __ballot_sync(FULL, v < n && __ldca(p + v) == giant);
          if (lane == 0 && v < n) A.bits[v >> 5] = b;
        }
      });
      if (!barrier()) return;
    }
  }
  // Labels: the smallest vertex of every tree, in q (the root itself is added
  // when read).
  vertices([&](int64_t v0) {
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int64_t v = v0 + j * 32 + lane;
      const int32_t root = v < n ? __ldca(p + v) : -1, root0 = __shfl_sync(FULL, root, 0);
      // (of the lanes under lane 0's root, lane 0 is the smallest vertex)
      if (v < root && (root != root0 || lane == 0)) offer(q, root, (int32_t)v);
    }
  });
  if (!barrier()) return;
  vertices([&](int64_t v0) {
    int32_t x[U];
    uint32_t y[U];
#pragma unroll
    for (int j = 0; j < U; ++j) x[j] = v0 + j * 32 + lane < n ? __ldca(p + v0 + j * 32 + lane) : 0;
#pragma unroll
    for (int j = 0; j < U; ++j) y[j] = __ldca(q + x[j]);
#pragma unroll
    for (int j = 0; j < U; ++j)
      if (v0 + j * 32 + lane < n) A.labels[v0 + j * 32 + lane] = (int32_t)min(y[j], (uint32_t)x[j]);
  });
  if (tid == 0) {
    A.host[1] = (unsigned)round + 1u;
    A.host[0] = 0u;
  }
}

}  // namespace

int components_pairs(int64_t n, int64_t m, const int2 *ends, int32_t *labels, int32_t *rounds, cudaStream_t s) {
  CcArgs A;
  std::memset(&A, 0, sizeof(A));
  A.n = n;
  A.m = m;
  A.ends = ends;
  A.labels = labels;
  int64_t want = ((m > n ? m : n) + BLOCK_SHARE - 1) / BLOCK_SHARE;
  if (want < 1 || (m <= ONE_BLOCK && n <= ONE_BLOCK)) want = 1;
  DeviceShare share(n, m);
  const int64_t cap = (int64_t)share.sms;
  const int blocks = (int)(want < cap ? want : cap);
  const int64_t warps = (int64_t)blocks * CW;
  A.es = page_shift(m, warps);
  A.vs = page_shift(n, warps);
  const size_t bit_bytes = (size_t)((n + 127) / 128) * 16;
  A.smem_bits = bit_bytes <= CC_BITS;
  A.few = n <= FEW && m >= 32 * n;
  size_t off = 0;
  auto place = [&](size_t bytes) {
    const size_t at = off;
    off = (off + bytes + 255) & ~(size_t)255;
    return at;
  };
  const size_t o_ctl = place(sizeof(CcCtrl)), o_p = place((size_t)(n + 1) * 4), o_q = place((size_t)(n + 1) * 4);
  const size_t o_deep = place(bit_bytes), o_bits = place(bit_bytes);
  const size_t o_list = place(((size_t)page_count(m, A.es) << A.es) * 8);
  int err = MSF_OK;
  char *base = (char *)pool_alloc(off, &err);
  if (err) return err;
  PoolBlock back{base};
  PinnedWords pin;
  if (int rc = pin.take(64)) return rc;
  Settle settle(s);
  pin.p[0] = 1u;
  A.ctl = (CcCtrl *)(base + o_ctl);
  A.p = (int32_t *)(base + o_p);
  A.q = (uint32_t *)(base + o_q);
  A.deep = (uint32_t *)(base + o_deep);
  A.bits = (uint32_t *)(base + o_bits);
  A.list = (int2 *)(base + o_list);
  A.host = pin.p;
  MSF_CK(cudaMemsetAsync(A.ctl, 0, sizeof(CcCtrl), s));
  size_t dyn = A.smem_bits ? bit_bytes : 0;
  if (A.few && dyn < FEW * 4) dyn = FEW * 4;
  cudaError_t e = cudaFuncSetAttribute(k_components, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CC_BITS);
  void *args[] = {&A};
  if (e == cudaSuccess)
    e = cudaLaunchCooperativeKernel((const void *)k_components, dim3((unsigned)blocks), dim3(CT), args, dyn, s);
  if (e == cudaErrorCooperativeLaunchTooLarge) {  // (a share of the device that holds fewer blocks)
    cudaGetLastError();
    MSF_CK(cudaStreamSynchronize(s));
    return SOLVE_NOT_RUN;
  }
  const cudaError_t e2 = cudaStreamSynchronize(s);
  settle.done = true;
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) return cuda_fail(e, "connected components");
  const volatile unsigned *st = pin.p;
  if (st[0] == 2u) return fail(MSF_ERR_ROUND_LIMIT, "round limit reached");
  if (st[0]) return fail(MSF_ERR_CHECK, "device consistency check failed");
  *rounds = (int32_t)st[1];
  return MSF_OK;
}

}  // namespace msf
