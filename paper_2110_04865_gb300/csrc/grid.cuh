// What the one-kernel solvers of a whole grid share: the barrier of all blocks,
// the pages in which edges and vertices are dealt to warps, relaxed accesses.
#pragma once

#include <cuda/atomic>

#include <cstdint>

namespace msf {

namespace {

__device__ __forceinline__ int ld_rel(const int32_t *a) {
  return cuda::atomic_ref<int, cuda::thread_scope_device>(*const_cast<int32_t *>(a)).load(cuda::memory_order_relaxed);
}
__device__ __forceinline__ void st_rel(int32_t *a, int v) {
  cuda::atomic_ref<int, cuda::thread_scope_device>(*a).store(v, cuda::memory_order_relaxed);
}

// Pages (see Pages) of 2^PAGE places at most, and smaller where a warp would get
// fewer than EVEN of them (its share is even to one page).  4096 graphs of 20 M
// edges: one range per warp 8.56 ms, pages of 128 7.0, by this rule 6.05, with
// EVEN 4 6.18, with longer pages 6.12; R-MAT and lattice graphs 1-5 % faster
// than with ranges.
constexpr int PAGE = 10, EVEN = 16;
inline int32_t page_shift(int64_t total, int64_t warps) {
  int32_t s = 7;
  while (s < PAGE && ((warps * EVEN) << (s + 1)) <= total) ++s;
  return s;
}
inline int64_t page_count(int64_t total, int32_t shift) { return (total + ((int64_t)1 << shift) - 1) >> shift; }

// Edges and vertices are dealt to the warps in pages: warp w of W takes pages
// w, w + W, ..., so that all warps work on one window of the arrays at a time
// (an input with locality -- a lattice, a batch -- then keeps the parents and
// minima it gathers in L2; with one contiguous range per warp every range's
// vicinity is live at once).  `at(i)` is the i-th of the warp's elements, in
// order; `cap` counts the places of its pages, `len` the elements below total.
struct Pages {
  uint32_t s, w, W, cap, len;
  __device__ Pages(int64_t total, int32_t shift, int64_t warp, int64_t warps)
      : s((uint32_t)shift), w((uint32_t)warp), W((uint32_t)warps) {
    const int64_t pages = (total + ((int64_t)1 << s) - 1) >> s;
    const int64_t mine = warp < pages ? (pages - warp + warps - 1) / warps : 0;
    cap = (uint32_t)(mine << s);
    len = cap;
    if (mine > 0 && (pages - 1) % warps == warp) len -= (uint32_t)((pages << s) - total);  // the last page
  }
  __device__ __forceinline__ uint32_t page(uint32_t i) const { return (i >> s) * W + w; }
  __device__ __forceinline__ int64_t at(uint32_t i) const {
    return ((int64_t)page(i) << s) + (i & ((1u << s) - 1u));
  }
};

// Barriers of a cooperative grid's blocks, with a sum on the way: an arrival adds 1
// above the block's addend, so the word that says that all have come also holds the
// sum (two words in turn: a block arrives at the next barrier but one only after all
// have read this one's).  An arrival takes the block's addend of the word's last
// barrier out again, so a sum is that of one barrier; until all have come it holds
// one addend of every block, this barrier's or the last one's: it neither borrows
// from the count above nor carries into it.  The wait is bounded.  One
// barrier is about 2 us of latency; what the words save is measured on whole calls,
// fences around the arrival, a counter and its read beside it before, this after:
// R-MAT 16 203 -> 173 us, R-MAT 20 500 -> 455, uniform m = 16 n 553 -> 505.
struct GridBarrier {  // in shared memory
  static constexpr int SHIFT = 46;  // arrivals above (1700 barriers of 152 blocks), sums below
  unsigned long long *word;         // [2], zero at the start
  unsigned *abort;                  // a wait ran out somewhere
  unsigned long long come[2], added[2], sum;  // arrivals awaited, the block's addends
  unsigned k, ok;
  __device__ void init(unsigned long long *w, unsigned *a) {  // (one thread; the block meets behind it)
    word = w;
    abort = a;
    come[0] = come[1] = added[0] = added[1] = 0;
    k = 0;
  }
  // All blocks meet; thread 0's `add` (below 2^38) summed up over them into `sum`.  False
  // (everywhere, sooner or later) when a wait ran out.
  __device__ bool meet(unsigned long long add = 0) {
    __syncthreads();
    if (threadIdx.x == 0) {
      if (gridDim.x == 1) {
        sum = add;
        ok = 1;
      } else {
        cuda::atomic_ref<unsigned long long, cuda::thread_scope_device> a(word[k & 1u]);
        cuda::atomic_ref<unsigned, cuda::thread_scope_device> ab(*abort);
        const unsigned long long all = come[k & 1u] += gridDim.x;
        // (released with the block's writes: it met before)
        a.fetch_add((1ull << SHIFT) + add - added[k & 1u], cuda::memory_order_release);
        added[k & 1u] = add;
        unsigned good = 0;
        for (unsigned it = 0; it < (1u << 25); ++it) {
          const unsigned long long v = a.load(cuda::memory_order_acquire);
          if ((v >> SHIFT) >= all) {
            sum = v & ((1ull << SHIFT) - 1ull);
            good = 1;
            break;
          }
          if ((it & 1023u) == 1023u && ab.load(cuda::memory_order_relaxed)) break;
        }
        if (!good) ab.store(1u, cuda::memory_order_relaxed);
        ++k;
        ok = good;
      }
    }
    __syncthreads();
    return ok != 0;
  }
};

// Edges e to e + 4 (or hi) of pairs of ends, 16-byte aligned.
__device__ __forceinline__ void load_pairs(const int2 *ends, int64_t e, int64_t hi, int4 &s, int4 &d) {
  if (e + 4 <= hi) {
    const int4 *q = reinterpret_cast<const int4 *>(ends + e);
    const int4 a = __ldcs(q), b = __ldcs(q + 1);
    s = make_int4(a.x, a.z, b.x, b.z);
    d = make_int4(a.y, a.w, b.y, b.w);
    return;
  }
  int32_t *x = &s.x, *y = &d.x;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (e + j < hi) {
      const int2 a = ends[e + j];
      x[j] = a.x;
      y[j] = a.y;
    }
}
}  // namespace

}  // namespace msf
