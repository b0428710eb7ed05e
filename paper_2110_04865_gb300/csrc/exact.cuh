// Device helpers shared by the solvers and the end-of-run kernels: the long
// accumulators of exact forest weights, thresholds of edge keys, and the
// expansion of the forest bitmap into mask bytes.
#pragma once

#include "internal.cuh"

namespace msf {

// float32: bins[b] accumulates the signed 24-bit significands of the weights
// whose (denormal-adjusted) biased exponent is b, so weight = sig * 2^(b-150);
// bin 0 counts +inf and bin 255 counts -inf.  uint32: bin 0 is the sum.
__device__ __forceinline__ void weight_bin(uint32_t ordw, int wtype, int *bin, long long *val) {
  if (wtype == MSF_U32) {
    *bin = 0;
    *val = (long long)ordw;
    return;
  }
  const uint32_t bits = (ordw & 0x80000000u) ? (ordw & 0x7fffffffu) : ~ordw;
  const uint32_t E = (bits >> 23) & 0xffu, M = bits & 0x7fffffu;
  const bool neg = bits >> 31;
  if (E == 255u) {
    *bin = neg ? 255 : 0;
    *val = 1;
    return;
  }
  const long long sig = E ? (long long)(M | 0x800000u) : (long long)M;
  *bin = E ? (int)E : 1;
  *val = neg ? -sig : sig;
}

// A block's long accumulators of float32 weights (weight_bin) in shared memory:
// 64-bit sums as two words, added with 32-bit shared atomics and a carry (a
// 64-bit shared atomic is a compare-and-swap loop, and a block's weights share
// few bins).  The low word is kept eight times, by lane, in eight banks: a
// warp's equal bins then serialise four deep instead of thirty-two.
struct BlockSums {
  unsigned lo[256][8], hi[256];
  __device__ void clear() {
    for (int i = threadIdx.x; i < 256 * 8; i += blockDim.x) lo[i >> 3][i & 7] = 0;
    for (int i = threadIdx.x; i < 256; i += blockDim.x) hi[i] = 0;
  }
  __device__ __forceinline__ void add(uint32_t ordw) {
    int bin;
    long long val;
    weight_bin(ordw, MSF_F32, &bin, &val);
    const unsigned v = (unsigned)val;
    const unsigned old = atomicAdd(&lo[bin][threadIdx.x & 7], v);
    const unsigned h = (unsigned)((unsigned long long)val >> 32) + (old + v < old ? 1u : 0u);
    if (h) atomicAdd(&hi[bin], h);
  }
  __device__ __forceinline__ void add_long(int bin, long long val) {
    const unsigned v = (unsigned)val;
    const unsigned old = atomicAdd(&lo[bin][0], v);
    const unsigned h = (unsigned)((unsigned long long)val >> 32) + (old + v < old ? 1u : 0u);
    if (h) atomicAdd(&hi[bin], h);
  }
  __device__ unsigned long long get(int b) const {
    unsigned long long t = (unsigned long long)hi[b] << 32;
#pragma unroll
    for (int k = 0; k < 8; ++k) t += lo[b][k];
    return t;
  }
};

// Unsigned big integer of 6 64-bit limbs.
struct Big {
  unsigned long long w[6];
};

__device__ __forceinline__ void big_add_shifted(Big &a, unsigned long long v, int sh) {
  // limbs below li get 0 with no carry; fixed trip counts keep the limbs in
  // registers
  const int li = sh >> 6, bo = sh & 63;
  const unsigned long long lo = v << bo;
  const unsigned long long hi = bo ? (v >> (64 - bo)) : 0ull;
  unsigned long long c = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const unsigned long long add = (i == li) ? lo : (i == li + 1 ? hi : 0ull);
    const unsigned long long s1 = a.w[i] + add;
    const unsigned long long c1 = s1 < add;
    const unsigned long long s2 = s1 + c;
    const unsigned long long c2 = s2 < c;
    a.w[i] = s2;
    c = c1 | c2;
  }
}

__device__ __forceinline__ int big_cmp(const Big &a, const Big &b) {
  for (int i = 5; i >= 0; --i) {
    if (a.w[i] != b.w[i]) return a.w[i] < b.w[i] ? -1 : 1;
  }
  return 0;
}

__device__ __forceinline__ void big_sub(Big &a, const Big &b) {  // a -= b, a >= b
  unsigned long long br = 0;
  for (int i = 0; i < 6; ++i) {
    const unsigned long long d1 = a.w[i] - b.w[i];
    const unsigned long long b1 = a.w[i] < b.w[i];
    const unsigned long long d2 = d1 - br;
    const unsigned long long b2 = d1 < br;
    a.w[i] = d2;
    br = b1 | b2;
  }
}


// Shifts that give 0 for shift counts of 64 or more.
__device__ __forceinline__ unsigned long long shl64(unsigned long long x, int s) { return s >= 64 ? 0ull : x << s; }
__device__ __forceinline__ unsigned long long shr64(unsigned long long x, int s) { return s >= 64 ? 0ull : x >> s; }

// Bits [lo, lo + 63] of a (lo >= 0).  Every limb is shifted into place (no
// limb is selected by a computed index, which would move a to local memory).
__device__ __forceinline__ unsigned long long big_window(const Big &a, int lo) {
  unsigned long long w = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const int d = i * 64 - lo;
    w |= d >= 0 ? shl64(a.w[i], d) : shr64(a.w[i], -d);
  }
  return w;
}

// Whether any bit below position `lo` is set.
__device__ __forceinline__ bool big_any_below(const Big &a, int lo) {
  bool any = false;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const int k = lo - i * 64;  // bits of limb i below lo
    const unsigned long long mk = k >= 64 ? ~0ull : (k <= 0 ? 0ull : (1ull << k) - 1ull);
    any = any || (a.w[i] & mk) != 0;
  }
  return any;
}

// Nearest double (ties to even) of (-1)^neg * a * 2^-149.
__device__ __forceinline__ double big_to_double(const Big &a, bool neg) {
  int h = -1;
#pragma unroll
  for (int i = 5; i >= 0; --i)
    if (h < 0 && a.w[i]) h = i * 64 + 63 - __clzll((long long)a.w[i]);
  if (h < 0) return 0.0;
  unsigned long long mant;
  int e2;  // value = mant * 2^e2
  if (h <= 52) {
    mant = a.w[0];
    e2 = -149;
  } else {
    // the 64 bits ending at h: top 53 are the significand, then the round
    // bit, then 10 bits that join the sticky bits below the window
    unsigned long long w;
    bool sticky;
    if (h >= 63) {
      w = big_window(a, h - 63);
      sticky = big_any_below(a, h - 63);
    } else {
      w = a.w[0] << (63 - h);
      sticky = false;
    }
    mant = w >> 11;
    const unsigned long long rb = (w >> 10) & 1ull;
    sticky = sticky || (w & 0x3ffull);
    e2 = h - 52 - 149;
    if (rb && (sticky || (mant & 1ull))) {
      mant += 1;
      if (mant == (1ull << 53)) {
        mant >>= 1;
        e2 += 1;
      }
    }
  }
  // normalize into [2^52, 2^53)
  while (mant < (1ull << 52)) {
    mant <<= 1;
    e2 -= 1;
  }
  const unsigned long long biased = (unsigned long long)(e2 + 52 + 1023);
  const unsigned long long bits = ((unsigned long long)neg << 63) | (biased << 52) | (mant & ((1ull << 52) - 1));
  return __longlong_as_double((long long)bits);
}

// a += b (six limbs; the sums of the accumulators stay far below 2^384)
__device__ __forceinline__ void big_add(Big &a, const Big &b) {
  unsigned long long c = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const unsigned long long s1 = a.w[i] + b.w[i];
    const unsigned long long c1 = s1 < b.w[i];
    const unsigned long long s2 = s1 + c;
    const unsigned long long c2 = s2 < c;
    a.w[i] = s2;
    c = c1 | c2;
  }
}

// Nearest double of (P - N) * 2^-149: |P - N| and its sign, one rounding;
// per-limb selects keep the limbs in registers.
__device__ __forceinline__ double round_difference(const Big &P, const Big &N) {
  const bool ge = big_cmp(P, N) >= 0;
  Big D, E;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    D.w[i] = ge ? P.w[i] : N.w[i];
    E.w[i] = ge ? N.w[i] : P.w[i];
  }
  big_sub(D, E);
  return big_to_double(D, !ge);
}

// Exact total of one graph from its long accumulators (bin 0: +inf count
// or, for u32 weights, the plain sum; bin 255: -inf count; bins 1..254:
// signed multiples of 2^(e-1)), rounded once to nearest even.
__device__ inline double combine_bins(const long long *b, int wtype) {
  if (wtype == MSF_U32) return __ull2double_rn((unsigned long long)b[0]);
  const bool pinf = b[0] > 0, ninf = b[255] > 0;
  if (pinf || ninf) {
    const unsigned long long bits = (pinf && ninf) ? 0x7ff8000000000000ull
                                    : (pinf ? 0x7ff0000000000000ull : 0xfff0000000000000ull);
    return __longlong_as_double((long long)bits);
  }
  Big P, N;
  for (int i = 0; i < 6; ++i) P.w[i] = N.w[i] = 0;
  for (int e = 1; e < 255; ++e) {
    const long long v = b[e];
    if (v > 0) big_add_shifted(P, (unsigned long long)v, e - 1);
    else if (v < 0) big_add_shifted(N, (unsigned long long)(-v), e - 1);
  }
  return round_difference(P, N);
}

// The same by a whole warp (every lane calls it; lane 0 gets the result):
// lane l adds bins 8l .. 8l+7 into its own pair of big integers, the pairs
// are summed across the warp, lane 0 rounds the difference once.
__device__ inline double combine_bins_warp(const long long *b, int wtype) {
  if (wtype == MSF_U32) return __ull2double_rn((unsigned long long)b[0]);
  const bool pinf = b[0] > 0, ninf = b[255] > 0;
  if (pinf || ninf) {
    const unsigned long long bits = (pinf && ninf) ? 0x7ff8000000000000ull
                                    : (pinf ? 0x7ff0000000000000ull : 0xfff0000000000000ull);
    return __longlong_as_double((long long)bits);
  }
  const int lane = threadIdx.x & 31;
  Big P, N;
#pragma unroll
  for (int i = 0; i < 6; ++i) P.w[i] = N.w[i] = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int e = 8 * lane + k;
    const long long v = (e >= 1 && e <= 254) ? b[e] : 0;
    if (v > 0) big_add_shifted(P, (unsigned long long)v, e - 1);
    else if (v < 0) big_add_shifted(N, (unsigned long long)(-v), e - 1);
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    Big P2, N2;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      P2.w[i] = __shfl_down_sync(0xffffffffu, P.w[i], off);
      N2.w[i] = __shfl_down_sync(0xffffffffu, N.w[i], off);
    }
    if (lane + off < 32) {
      big_add(P, P2);
      big_add(N, N2);
    }
  }
  return round_difference(P, N);
}

// The rank among `samples` evenly spread ones whose key takes about light * n of m
// edges.  A low rank is a matter of luck -- the fourth of 256 samples may leave a
// quarter of the edges meant, whose forest holds few of the others back -- so with
// many edges a vertex it is not below 2 * low or three edges a vertex, and not below
// low unless that makes 32 a vertex.  Mean of 8 to 24 seeds in us, without / with:
// 40 graphs of 2000 vertices and 2^19 edges 2258 / 443, 152 of 1000 and 60 000 278 /
// 133, 100 of 2000 and 10^5 399 / 165; one of 10^5 and 16 M 396 / 307.
// (In float: a block's warp 0 waits for it, and double operations were 2 us of the
// 95 of 4096 vertices and 32 768 edges.)
__host__ __device__ inline int light_rank(double light, int64_t n, int64_t m, int samples, int low) {
  const float per = (float)n / (float)m * (float)samples;  // samples to an edge a vertex
  float least = 32.f * per < (float)low ? 32.f * per : (float)low;
  if (least < 2.f) least = 2.f;
  float want = 3.f * per < 2.f * (float)low ? 3.f * per : 2.f * (float)low;
  if (want < least) want = least;
  const float rank = (float)light * per;
  return (int)(rank > want ? rank : want);
}

// Whether a weight lies below a threshold key (weight tw, edge index te, te a
// multiple of 128): one comparison per edge, with the edges of a batch of 128
// all on one side of te.
template <bool F32>
struct Limit {
  uint32_t at, under;  // largest weight below the threshold, for edges before and from te
  int64_t te;
  bool none;           // no weight lies below it from te on
  uint32_t lim;
  bool ok;
  __device__ Limit(unsigned long long T) {
    const uint32_t tw = (uint32_t)(T >> 32);
    te = (int64_t)(uint32_t)T == 0xffffffffll ? (int64_t)1 << 40 : (int64_t)(uint32_t)T;
    at = tw;
    none = tw == 0;
    under = tw - (none ? 0u : 1u);
    if (F32) {  // the comparison is of floats (NaN: false)
      at = from_ord(at);
      under = none ? 0x7fffffffu : from_ord(under);
    }
  }
  __device__ static uint32_t from_ord(uint32_t o) {
    uint32_t b = (o & 0x80000000u) ? o & 0x7fffffffu : ~o;
    if (b == 0x80000000u) b = 0x80000001u;  // (-0 is ordered as +0: below +0 are the negative weights)
    return (b << 1) > 0xff000000u ? ((b >> 31) ? 0x7fffffffu : 0x7f800000u) : b;
  }
  __device__ __forceinline__ void batch(int64_t e) {  // the batch of edges from e on
    const bool before = e < te;
    lim = before ? at : under;
    ok = F32 || before || !none;
  }
  __device__ __forceinline__ bool below(uint32_t w, int64_t e) const {  // of an edge on its own
    if (F32) return __uint_as_float(w) <= __uint_as_float(e < te ? at : under);
    return e < te ? w <= at : (w <= under && !none);
  }
  __device__ __forceinline__ bool below(uint32_t w) const {
    return F32 ? __uint_as_float(w) <= __uint_as_float(lim) : (w <= lim && ok);
  }
};

// Four consecutive edges from index i on, of the edges [lo, hi) of the arrays
// at src, dst, w; the others become self-loops of vertex 0.  vec: the arrays
// are 16-byte aligned and i is a multiple of four.
struct EdgeQuad {
  int4 s, d;
  uint4 w;
};
template <bool W>
__device__ __forceinline__ EdgeQuad edge_quad(const int32_t *src, const int32_t *dst, const uint32_t *w, bool vec, int i,
                                            int lo, int hi) {
  EdgeQuad q;
  q.s = q.d = make_int4(0, 0, 0, 0);
  q.w = make_uint4(0u, 0u, 0u, 0u);
  if (vec && i >= lo && i + 4 <= hi) {
    q.s = *reinterpret_cast<const int4 *>(src + i);
    q.d = *reinterpret_cast<const int4 *>(dst + i);
    if (W) q.w = *reinterpret_cast<const uint4 *>(w + i);
    return q;
  }
  int32_t *s = &q.s.x, *d = &q.d.x;
  uint32_t *v = &q.w.x;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (i + j >= lo && i + j < hi) {
      s[j] = src[i + j];
      d[j] = dst[i + j];
      if (W) v[j] = w[i + j];
    }
  return q;
}

// The same from pairs of ends (16-byte aligned, as w), edges [i, hi) of four.
__device__ __forceinline__ EdgeQuad pair_quad(const int2 *ends, const uint32_t *w, int i, int hi) {
  EdgeQuad q;
  q.s = q.d = make_int4(0, 0, 0, 0);
  q.w = make_uint4(0u, 0u, 0u, 0u);
  if (i + 4 <= hi) {
    const int4 a = reinterpret_cast<const int4 *>(ends + i)[0], b = reinterpret_cast<const int4 *>(ends + i)[1];
    q.s = make_int4(a.x, a.z, b.x, b.z);
    q.d = make_int4(a.y, a.w, b.y, b.w);
    q.w = *reinterpret_cast<const uint4 *>(w + i);
    return q;
  }
  int32_t *s = &q.s.x, *d = &q.d.x;
  uint32_t *v = &q.w.x;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (i + j < hi) {
      const int2 uv = ends[i + j];
      s[j] = uv.x;
      d[j] = uv.y;
      v[j] = w[i + j];
    }
  return q;
}

// Batches of 128 edges [lo, hi) through two register buffers in turn: a buffer
// is loaded again once its batch is done, while the other's is worked on, and
// none is copied to the other.
template <class Q, class Load, class Body>
__device__ __forceinline__ void stream2(int lo, int hi, Load load, Body body) {
  Q a = load(lo), b = load(lo + 128);
  for (int k = lo; k < hi; k += 256) {
    body(a, k);
    a = load(k + 256);
    if (k + 128 < hi) body(b, k + 128);
    b = load(k + 384);
  }
}

// 16 mask bytes from 16 bits: byte j = bit j (each nibble spread to the low
// bits of four bytes by one multiplication: its copies at shifts 0, 7, 14
// and 21 do not overlap, and bit j of the nibble lands on bit 8j).
__device__ __forceinline__ uint4 spread16(uint32_t v) {
  constexpr uint32_t MUL = 0x00204081u, LOW = 0x01010101u;
  return make_uint4(((v & 0xfu) * MUL) & LOW, (((v >> 4) & 0xfu) * MUL) & LOW, (((v >> 8) & 0xfu) * MUL) & LOW,
                    (((v >> 12) & 0xfu) * MUL) & LOW);
}
// bits [e, e + 16) of the bitmap (the bitmap has a zero word past the end)
__device__ __forceinline__ uint32_t bits16(const uint32_t *bits, int64_t e) {
  const int64_t i = e >> 5;
  const uint32_t o = (uint32_t)(e & 31);
  const uint64_t w = (uint64_t)bits[i] | ((uint64_t)bits[i + 1] << 32);
  return (uint32_t)(w >> o) & 0xffffu;
}
}  // namespace msf
