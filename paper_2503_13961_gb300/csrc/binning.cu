// Tile binning and the (tile, depth) sort of the Gaussians, and the per-tile
// boundary-point lists sorted by primitive id (Sec. 3.2, "Rendering
// Acceleration": precomputed tile range of each boundary point, per-tile
// lists sorted by ID so that a binary search finds a primitive's points).
//
// The sort is a most-significant-digit radix sort of the key (tile, depth,
// index): the first digit is the whole tile id (a counting sort: per-tile
// counts from the generation pass, an exclusive scan, one scatter), the
// remaining 64 bits (36-bit depth key = FP32 depth bits and 5 finer bits,
// 27-bit Gaussian index) are sorted inside each tile by a network held in
// registers. Keys are unique, so the order is fully determined.
// Boundary keys are (primitive, boundary index).
#include <cooperative_groups.h>

#include <algorithm>

#include "bgt_internal.cuh"

namespace bgt {

namespace {

// Scans of the per-tile and per-primitive counts: one launch of one cluster of
// thread blocks. Every block sums its range of the counts, the blocks read
// each other's sums from distributed shared memory behind one cluster
// barrier, and each then scans its range; 8 blocks above kScanOne elements,
// one below (a barrier less). No block waits for another but at that barrier.
// A reduce, a scan of the block sums and a down-sweep as launches of their own took
// ~10 us per array in the small calls, where every launch of the serial chain
// costs 2-4 us whatever it does.
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanChunk = kScanThreads * kScanItems;
constexpr int kScanOne = 2 * kScanChunk;
constexpr int kScanCluster = 8;

// warp-inclusive sums of two values
__device__ __forceinline__ void warp_scan2(long long &a, long long &b) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long x = __shfl_up_sync(0xffffffffu, a, o), y = __shfl_up_sync(0xffffffffu, b, o);
    if (lane >= o) {
      a += x;
      b += y;
    }
  }
}

// exclusive scan over the block of two values per thread; tot: the block's sums
__device__ inline void block_scan2(long long &a, long long &b, longlong2 &tot, longlong2 *s_warp) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const long long a0 = a, b0 = b;
  warp_scan2(a, b);
  __syncthreads();  // s_warp is free
  if (lane == 31) s_warp[wp] = make_longlong2(a, b);
  __syncthreads();
  const longlong2 v = s_warp[lane];  // 32 warps
  longlong2 inc = v;
  warp_scan2(inc.x, inc.y);
  tot.x = __shfl_sync(0xffffffffu, inc.x, 31);
  tot.y = __shfl_sync(0xffffffffu, inc.y, 31);
  a += __shfl_sync(0xffffffffu, inc.x - v.x, wp) - a0;
  b += __shfl_sync(0xffffffffu, inc.y - v.y, wp) - b0;
}

// Exclusive prefix sums of two count arrays (16-byte aligned, as the outputs), the totals last. Returns
// the totals on every thread.
template <int CL>
__device__ inline longlong2 scan_both(const int *in0, long long *out0, const int *in1, long long *out1, int n) {
  __shared__ longlong2 s_warp[32], s_sum;
  const int4 *p0 = reinterpret_cast<const int4 *>(in0), *p1 = reinterpret_cast<const int4 *>(in1);
  // this block's range [lo, hi), a multiple of kScanChunk long but for the last
  const int chunks = (n + kScanChunk - 1) / kScanChunk, per = (chunks + CL - 1) / CL * kScanChunk;
  const int lo = min((int)blockIdx.x * per, n), hi = min(lo + per, n);
  longlong2 run = make_longlong2(0, 0);
  if constexpr (CL > 1) {
    namespace cg = cooperative_groups;
    long long a = 0, b = 0;
#pragma unroll 4
    for (int i = (lo >> 2) + threadIdx.x; i < hi >> 2; i += kScanThreads) {
      const int4 x = p0[i], y = p1[i];
      a += ((long long)x.x + x.y) + ((long long)x.z + x.w);
      b += ((long long)y.x + y.y) + ((long long)y.z + y.w);
    }
    if ((int)threadIdx.x < (hi & 3) && hi > lo) {
      a += in0[(hi & ~3) + threadIdx.x];
      b += in1[(hi & ~3) + threadIdx.x];
    }
    longlong2 sum;
    block_scan2(a, b, sum, s_warp);
    if (threadIdx.x == 0) s_sum = sum;
    const cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    for (int k = 0; k < (int)blockIdx.x; k++) {
      const longlong2 o = *cl.map_shared_rank(&s_sum, k);
      run.x += o.x;
      run.y += o.y;
    }
    cl.sync();  // no block leaves while its sum may still be read
  }
  for (int base = lo; base < hi; base += kScanChunk) {
    const int i = base + (int)threadIdx.x * kScanItems;
    int4 x = make_int4(0, 0, 0, 0), y = x;
    if (i + 3 < hi) {
      x = p0[i >> 2];
      y = p1[i >> 2];
    } else {
      if (i < hi) { x.x = in0[i]; y.x = in1[i]; }
      if (i + 1 < hi) { x.y = in0[i + 1]; y.y = in1[i + 1]; }
      if (i + 2 < hi) { x.z = in0[i + 2]; y.z = in1[i + 2]; }
    }
    long long a = ((long long)x.x + x.y) + ((long long)x.z + x.w), b = ((long long)y.x + y.y) + ((long long)y.z + y.w);
    longlong2 tot;
    block_scan2(a, b, tot, s_warp);
    a += run.x;
    b += run.y;
    const long long sa[4] = {a, a + x.x, a + x.x + x.y, a + x.x + x.y + x.z};
    const long long sb[4] = {b, b + y.x, b + y.x + y.y, b + y.x + y.y + y.z};
    if (i + 3 < hi) {
      longlong2 *o0 = reinterpret_cast<longlong2 *>(out0 + i), *o1 = reinterpret_cast<longlong2 *>(out1 + i);
      o0[0] = make_longlong2(sa[0], sa[1]);
      o0[1] = make_longlong2(sa[2], sa[3]);
      o1[0] = make_longlong2(sb[0], sb[1]);
      o1[1] = make_longlong2(sb[2], sb[3]);
    } else {
#pragma unroll
      for (int k = 0; k < 3; k++)
        if (i + k < hi) {
          out0[i + k] = sa[k];
          out1[i + k] = sb[k];
        }
    }
    run.x += tot.x;
    run.y += tot.y;
  }
  if (hi == n && lo < n && threadIdx.x == 0) {  // the block of the last element holds the totals
    out0[n] = run.x;
    out1[n] = run.y;
  }
  return run;
}

template <int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(kScanThreads)
    k_scan_pair(int *in0, long long *out0, int *in1, long long *out1, int n, bool clear) {
  chained();
  scan_both<CL>(in0, out0, in1, out1, n);
  if (!clear) return;
  // every count of the block's range was last read before its last block barrier, but for the final chunk's
  __syncthreads();
  const int chunks = (n + kScanChunk - 1) / kScanChunk, per = (chunks + CL - 1) / CL * kScanChunk;
  const int lo = min((int)blockIdx.x * per, n), hi = min(lo + per, n);
  for (int i = lo + (int)threadIdx.x; i < hi; i += kScanThreads) in0[i] = in1[i] = 0;
}

// Tile list starts (exclusive sums of the Gaussian and boundary counts) and the
// capacity check, by the block that holds the last tile
template <int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(kScanThreads) k_tile_scan(Params p, Work w) {
  chained();
  const longlong2 total = scan_both<CL>(w.g_tcount, w.g_tstart, w.b_tcount, w.b_tstart, p.tiles);
  const int chunks = (p.tiles + kScanChunk - 1) / kScanChunk, per = (chunks + CL - 1) / CL * kScanChunk;
  if ((int)blockIdx.x == (p.tiles - 1) / per && threadIdx.x == 0) {
    w.counters[kK] = (int)min(total.x, 0x7fffffffll);
    w.counters[kKb] = (int)min(total.y, 0x7fffffffll);
    if (total.x > p.max_pairs) atomicOr(w.status, kStatusPairOverflow);
    if (total.y > p.max_bpairs) atomicOr(w.status, kStatusBoundaryOverflow);
  }
}

// per-tile descriptor, so that the blending kernels read two records instead
// of searching the view offsets and reading the list starts: [2t] geometry,
// [2t + 1] (Gaussian list start, length, boundary list start, length); an
// overflowed list (its slots were not all written) has length 0
__device__ inline void tile_descriptor(const Params &p, const Work &w, int t) {
  const int view = find_view(w.view_tile_off, p.V, t);
  const View &vw = w.views[view];
  const int lt = t - vw.tile_off;
  const int ty = lt / vw.tiles_x, tx = lt - ty * vw.tiles_x;
  w.tile_desc[2 * t] = make_int4(view, (int)((unsigned)(tx * p.tile) | ((unsigned)(ty * p.tile) << 16)),
                                 (int)((unsigned)vw.W | ((unsigned)vw.H << 16)), vw.pix_off);
  const bool g_over = w.g_tstart[p.tiles] > p.max_pairs, b_over = w.b_tstart[p.tiles] > p.max_bpairs;
  const long long gs = w.g_tstart[t], bs = w.b_tstart[t];
  w.tile_desc[2 * t + 1] = make_int4(g_over ? 0 : (int)gs, g_over ? 0 : (int)(w.g_tstart[t + 1] - gs),
                                     b_over ? 0 : (int)bs, b_over ? 0 : (int)(w.b_tstart[t + 1] - bs));
}

// a slot in tile t's segment: the active lanes of the warp that want one in
// the same tile share one atomic (consecutive Gaussians mostly share tiles);
// the order inside a segment is set by the sort that follows
__device__ __forceinline__ int tile_slot(int *fill, int t) {
  const int lane = threadIdx.x & 31;
  const unsigned peers = __match_any_sync(__activemask(), t);
  const int leader = __ffs(peers) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(fill + t, __popc(peers));
  base = __shfl_sync(peers, base, leader);
  return base + __popc(peers & ((1u << lane) - 1u));
}

__device__ inline void emit_rect(unsigned long long *keys, int *fill, const long long *start, long long cap,
                                 int tile_off, int tiles_x, uint2 rect, unsigned long long hi,
                                 unsigned lo) {
  const int x0 = rect.x & 0xffff, y0 = rect.x >> 16, x1 = rect.y & 0xffff, y1 = rect.y >> 16;
  for (int ty = y0; ty <= y1; ty++)
    for (int tx = x0; tx <= x1; tx++) {
      const int t = tile_off + ty * tiles_x + tx;
      const long long pos = start[t] + tile_slot(fill, t);
      if (pos >= 0 && pos < cap) keys[pos] = hi | (unsigned long long)lo;
    }
}

// the pair keys, unsorted, into the second halves of the key arrays (the sort
// writes the first), and the tiles' descriptors
__global__ void k_emit(Params p, Work w) {
  chained();
  const int F = w.counters[kF], Nb = w.counters[kNb];
  const int stride = gridDim.x * blockDim.x;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < p.tiles; t += stride) tile_descriptor(p, w, t);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < F; i += stride) {
    const uint2 rect = w.g_rect[i];
    if ((rect.x & 0xffff) > (rect.y & 0xffff)) continue;
    const View *vw = w.views + w.g_view[i];
    const unsigned long long dkey =
        ((unsigned long long)__float_as_uint(w.g_depth[i]) << 5) | (unsigned long long)w.g_dsub[i];
    emit_rect(w.gkeys + p.max_pairs, w.g_tfill, w.g_tstart, p.max_pairs, __ldg(&vw->tile_off), __ldg(&vw->tiles_x),
              rect, dkey << kIndexBits, (unsigned)i);
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Nb; i += stride) {
    const uint2 rect = w.b_rect[i];
    if ((rect.x & 0xffff) > (rect.y & 0xffff)) continue;
    const View *vw = w.views + w.b_view[i];
    emit_rect(w.bkeys + p.max_bpairs, w.b_tfill, w.b_tstart, p.max_bpairs, __ldg(&vw->tile_off), __ldg(&vw->tiles_x),
              rect, (unsigned long long)(unsigned)w.b_prim[i] << 32, (unsigned)i);
  }
}

// ---------------------------------------------------------------------------
// per-tile sort
// ---------------------------------------------------------------------------
constexpr int kSortThreads = 128;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kRunCap = 512;                    // keys one warp sorts in registers (16 per lane)
constexpr int kWarpSortCap = 2 * kRunCap;       // keys one warp sorts: two such runs, merged
constexpr int kSortCap = kSortWarps * kWarpSortCap;  // keys one block sorts in shared memory
constexpr int kLongCap = 8 * kSortCap;               // keys one block sorts as runs of kSortCap, merged
constexpr int kFullKeys = 1 << 30;              // flag of a listed segment: its order needs all key bits

// position of key i in shared memory: one key of padding per 16, so that lanes
// writing runs of consecutive keys (16 apart, say) hit distinct banks
__host__ __device__ constexpr int padded(int i) { return i + (i >> 4); }
constexpr int kWarpWords = padded(kWarpSortCap);  // a warp's words; every warp and block holds them twice
constexpr int kSortBigSmem = 2 * kSortWarps * kWarpWords * (int)sizeof(unsigned);
static_assert(kSortBigSmem >= padded(kSortCap) * (int)sizeof(unsigned long long), "the keys of a segment fit as well");

__device__ __forceinline__ void key_order(unsigned &a, unsigned &b) {
  const unsigned lo = min(a, b);
  b = max(a, b);
  a = lo;
}

__device__ __forceinline__ void take_order(unsigned &k, unsigned o, bool upper) {
  const unsigned lo = min(k, o), hi = max(k, o);
  k = upper ? hi : lo;
}

__device__ __forceinline__ void take_order(unsigned long long &k, unsigned long long o, bool upper) {
  k = (o < k) != upper ? o : k;
}

__device__ __forceinline__ void key_order(unsigned long long &a, unsigned long long &b) {
  const bool swap = b < a;
  const unsigned long long lo = swap ? b : a;
  b = swap ? a : b;
  a = lo;
}

// Batcher's odd-even merge network (1968) of E keys in one lane's registers:
// stages p = 1, 2, .. E / 2, in each distances q = p, p / 2, .. 1
template <int E, int P, int Q, class Key>
__device__ __forceinline__ void odd_even_stage(Key (&k)[E]) {
#pragma unroll
  for (int i = Q % P; i + Q < E; i++)
    if ((i - Q % P) % (2 * Q) < Q && i / (2 * P) == (i + Q) / (2 * P)) key_order(k[i], k[i + Q]);
  if constexpr (Q > 1) odd_even_stage<E, P, Q / 2>(k);
  else if constexpr (2 * P < E) odd_even_stage<E, 2 * P, 2 * P>(k);
}

// bitonic merge of a lane's keys: distances J, J / 2, .. 1
template <int E, int J, class Key>
__device__ __forceinline__ void halving_steps(Key (&k)[E]) {
#pragma unroll
  for (int e = 0; e < E; e++)
    if (!(e & J)) key_order(k[e], k[e | J]);
  if constexpr (J > 1) halving_steps<E, J / 2>(k);
}

// Sort of 32 E keys by one warp in registers, ascending, key i in lane i / E,
// register i % E: every lane sorts its own keys (no shuffles), then lane groups of 2, 4, .. 32 merge
// bitonically: a first step against the mirrored position of the other half
// (so that every comparison is ascending), then halving distances, by
// shuffles down to one lane and in registers inside it. 15 shuffle steps at
// any E; neighbouring keys in one lane is what keeps them this few (keys 32
// apart per lane need 35 at 512 keys).
template <int E, class Key>
__device__ __forceinline__ void warp_sort_regs(Key (&k)[E], int lane) {
  if constexpr (E > 1) odd_even_stage<E, 1, 1>(k);
#pragma unroll 1
  for (int s = 2; s <= 32; s <<= 1) {
    {
      const bool upper = lane & (s >> 1);
#pragma unroll
      for (int e = 0; e < (E + 1) / 2; e++) {
        const Key oa = __shfl_xor_sync(0xffffffffu, k[E - 1 - e], s - 1);
        if (E > 1) {
          const Key ob = __shfl_xor_sync(0xffffffffu, k[e], s - 1);
          take_order(k[E - 1 - e], ob, upper);
        }
        take_order(k[e], oa, upper);
      }
    }
#pragma unroll 1
    for (int j = s >> 2; j >= 1; j >>= 1) {
      const bool upper = lane & j;
#pragma unroll
      for (int e = 0; e < E; e++) take_order(k[e], __shfl_xor_sync(0xffffffffu, k[e], j), upper);
    }
    if constexpr (E > 1) halving_steps<E, E / 2>(k);
  }
}

// Stable block-wide LSD radix sort (8-bit digits) of the segment `keys` in
// global memory into `out`, for segments larger than the shared-memory
// capacity; `keys` is scratch afterwards. Digits that are equal across the
// whole segment are skipped.
__device__ void radix_global(unsigned long long *keys, unsigned long long *out, int n, int *s_hist,
                             int *s_base, int *s_wcnt, unsigned long long *s_red) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = kSortThreads / 32;
  // OR / AND over the segment to find constant digits
  unsigned long long vor = 0ull, vand = ~0ull;
  for (int i = threadIdx.x; i < n; i += kSortThreads) {
    vor |= keys[i];
    vand &= keys[i];
  }
  for (int o = 16; o > 0; o >>= 1) {
    vor |= __shfl_xor_sync(0xffffffffu, vor, o);
    vand &= __shfl_xor_sync(0xffffffffu, vand, o);
  }
  if (lane == 0) { s_red[wp] = vor; s_red[nw + wp] = vand; }
  __syncthreads();
  vor = 0ull; vand = ~0ull;
  for (int i = 0; i < nw; i++) { vor |= s_red[i]; vand &= s_red[nw + i]; }
  __syncthreads();
  const unsigned long long varying = vor ^ vand;
  unsigned long long *src = keys, *dst = out;
  for (int shift = 0; shift < 64; shift += 8) {
    if (((varying >> shift) & 0xffull) == 0ull) continue;
    for (int d = threadIdx.x; d < 256; d += kSortThreads) s_hist[d] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kSortThreads) atomicAdd(&s_hist[(src[i] >> shift) & 0xff], 1);
    __syncthreads();
    if (threadIdx.x == 0) {
      int run = 0;
      for (int d = 0; d < 256; d++) { s_base[d] = run; run += s_hist[d]; }
    }
    for (int d = threadIdx.x; d < nw * 256; d += kSortThreads) s_wcnt[d] = 0;
    __syncthreads();
    for (int chunk = 0; chunk < n; chunk += kSortThreads) {
      const int i = chunk + threadIdx.x;
      const bool valid = i < n;
      const unsigned long long key = valid ? src[i] : 0ull;
      const int dig = valid ? (int)((key >> shift) & 0xff) : 256 + wp;
      const unsigned peers = __match_any_sync(0xffffffffu, dig);
      const int rank = __popc(peers & ((1u << lane) - 1u));
      if (valid && rank == 0) s_wcnt[wp * 256 + dig] = __popc(peers);
      __syncthreads();
      if (valid) {
        int pos = s_base[dig] + rank;
        for (int q = 0; q < wp; q++) pos += s_wcnt[q * 256 + dig];
        dst[pos] = key;
      }
      __syncthreads();
      for (int d = threadIdx.x; d < 256; d += kSortThreads) {
        int add = 0;
        for (int q = 0; q < nw; q++) { add += s_wcnt[q * 256 + d]; s_wcnt[q * 256 + d] = 0; }
        s_base[d] += add;
      }
      __syncthreads();
    }
    unsigned long long *t = src; src = dst; dst = t;
  }
  if (src != out)
    for (int i = threadIdx.x; i < n; i += kSortThreads) out[i] = src[i];
  __syncthreads();
}

__device__ inline void segment_bounds(const Params &p, const Work &w, int item, bool &bnd, long long &s0,
                                      long long &s1) {
  bnd = item >= p.tiles;
  const int tile = bnd ? item - p.tiles : item;
  const long long *start = bnd ? w.b_tstart : w.g_tstart;
  const long long cap = bnd ? p.max_bpairs : p.max_pairs;
  s0 = start[tile];
  s1 = start[tile + 1];
  s0 = s0 < 0 ? 0 : (s0 > cap ? cap : s0);
  s1 = s1 < s0 ? s0 : (s1 > cap ? cap : s1);
}

// a sorted key to its place in the list; a boundary key's record beside it
__device__ __forceinline__ void store_sorted(const Work &w, bool bnd, long long at, unsigned long long key) {
  if (!bnd) {
    w.gkeys[at] = key;
    return;
  }
  w.bkeys[at] = key;
  w.bl_prim[at] = (int)(key >> 32);
  w.bl_rec[at] = w.bR[(unsigned)(key & 0xffffffffu)];
}

// How the 64-bit keys of one segment are sorted as 32-bit words, which one
// compare-exchange of the network moves in two instructions instead of six (and
// the network's code, a third of the size, stays in the instruction cache).
//   Exact words: (primitive or depth key - least) << index bits | (index -
//   least), the key itself shortened, when both ranges fit 31 bits together.
//   Boundary keys have no other; of the Gaussian keys it is those of a surface at
//   one depth, whose ties no position resolves: a wall that faces eight 1600 x
//   1200 views (58 M pairs) took the binning 10.1 ms when its lists ended on all key bits, now 0.91.
//   Gaussian keys otherwise: the depth key less the least FP32 depth of the segment,
//   cut to its upper bits, with the key's position in the segment below them.
//   Depths that differ only in the cut bits, and ties of depth, may leave
//   neighbours out of order: words that agree above their positions are
//   exchanged by their full keys (groups of up to 3 on the room's tiles).
// Segments that fit neither are sorted on all key bits.
struct WordForm {
  unsigned hi0, lo0;   // least high word and index
  int low, down, up;   // key bits below the primitive or depth key, its bits cut off, word bits below it
  bool exact, ok;
};

// least and greatest high word and index of a segment
struct KeyRange {
  unsigned hi0, hi1, lo0, lo1;
};

__device__ __forceinline__ KeyRange key_range(const unsigned long long *keys, int n, int first, int step) {
  KeyRange r{0xffffffffu, 0u, 0xffffffffu, 0u};
  for (int i = first; i < n; i += step) {
    const unsigned long long k = keys[i];
    const unsigned hi = (unsigned)(k >> 32), lo = (unsigned)(k & kIndexMask);
    r.hi0 = min(r.hi0, hi);
    r.hi1 = max(r.hi1, hi);
    r.lo0 = min(r.lo0, lo);
    r.lo1 = max(r.lo1, lo);
  }
  r.hi0 = __reduce_min_sync(0xffffffffu, r.hi0);
  r.hi1 = __reduce_max_sync(0xffffffffu, r.hi1);
  r.lo0 = __reduce_min_sync(0xffffffffu, r.lo0);
  r.lo1 = __reduce_max_sync(0xffffffffu, r.lo1);
  return r;
}

// n: keys of the segment
__device__ __forceinline__ WordForm word_form(const KeyRange &r, bool bnd, int n) {
  WordForm f;
  f.hi0 = r.hi0;
  f.lo0 = r.lo0;
  f.low = bnd ? 32 : kIndexBits;
  const unsigned span = r.hi1 - r.hi0;
  const bool narrow = span < (1u << 27);  // the depth key less (hi0 << 5) fits 32 bits
  const int bits = bnd ? 32 - __clz((int)span) : narrow ? 32 - __clz((int)((span << 5) | 31u)) : 32;
  const int index_bits = 32 - __clz((int)(r.lo1 - r.lo0));
  const int pos_bits = max(5, 32 - __clz(n));  // one more position than keys for the padding word
  f.exact = index_bits + bits <= 31;
  f.ok = f.exact || (!bnd && narrow);
  f.down = f.exact ? 0 : max(0, bits - (32 - pos_bits));
  f.up = f.exact ? index_bits : pos_bits;
  return f;
}

__device__ __forceinline__ unsigned key_word(const WordForm &f, unsigned long long key, int pos) {
  const unsigned rank = __funnelshift_rc((unsigned)key, (unsigned)(key >> 32) - f.hi0, f.low);
  return ((rank >> f.down) << f.up) | (f.exact ? (unsigned)(key & kIndexMask) - f.lo0 : (unsigned)pos);
}

__device__ __forceinline__ unsigned long long word_key(const WordForm &f, const unsigned long long *keys, unsigned word) {
  const unsigned lo = word & ((1u << f.up) - 1u);
  if (!f.exact) return keys[lo];
  return ((unsigned long long)f.hi0 << 32) + ((unsigned long long)(word >> f.up) << f.low) + (lo + f.lo0);
}

constexpr int kFixPasses = 8;  // rounds of neighbour exchanges before a list is sorted on all bits

struct Padded {
  __device__ int operator()(int i) const { return padded(i); }
};

// One round of exchanges (even, then odd neighbours) among the sorted words of a
// Gaussian list that agree above their position bits, by the full keys; true
// if any moved. SYNC separates the two halves and ends the round. Word i is at s[at(i)].
template <class At, class Sync>
__device__ __forceinline__ bool exchange_ties(const unsigned long long *keys, unsigned *s, At at, int n, int pos_bits,
                                              int first, int step, Sync sync) {
  const unsigned mask = (1u << pos_bits) - 1u;
  bool moved = false;
  for (int odd = 0; odd < 2; odd++) {
    for (int i = 2 * first + odd; i + 1 < n; i += 2 * step) {
      const unsigned a = s[at(i)], b = s[at(i + 1)];
      if (((a ^ b) >> pos_bits) == 0u && keys[b & mask] < keys[a & mask]) {
        s[at(i)] = b;
        s[at(i + 1)] = a;
        moved = true;
      }
    }
    sync();
  }
  return moved;
}

// The words of keys[0, n), n <= 32 E, with positions from `first` on, sorted by one warp into s (padded
// positions from `first` on). Not inlined: the two runs of a segment share the
// code of a size, which has to stay in the instruction cache (a form of 32
// words per lane beside it made the fetches the first stall).
template <int E>
__device__ __noinline__ void warp_sort_run(const unsigned long long *keys, unsigned *s, WordForm f, int first, int n) {
  const int lane = threadIdx.x & 31;
  unsigned k[E];
#pragma unroll
  for (int e = 0; e < E; e++) {
    const int i = e * 32 + lane;
    k[e] = i < n ? key_word(f, keys[i], first + i) : 0xffffffffu;  // padding: last in any order
  }
  warp_sort_regs<E>(k, lane);
#pragma unroll
  for (int e = 0; e < E; e++)
    if (lane * E + e < n) s[padded(first + lane * E + e)] = k[e];
}

__device__ __forceinline__ void sort_run(const unsigned long long *keys, unsigned *s, const WordForm &f, int first,
                                         int n) {
  if (n <= 32) warp_sort_run<1>(keys, s, f, first, n);
  else if (n <= 64) warp_sort_run<2>(keys, s, f, first, n);
  else if (n <= 128) warp_sort_run<4>(keys, s, f, first, n);
  else if (n <= 256) warp_sort_run<8>(keys, s, f, first, n);
  else warp_sort_run<16>(keys, s, f, first, n);
}

// Outputs [d0, d1) of the merge of the sorted runs s[a, a + na) and s[b, b + nb)
// (distinct words) into out from position o on: the split of the first output
// by binary search along its diagonal (merge path, Green et al. 2012), then
// one word at a time.
__device__ __forceinline__ void merge_part(const unsigned *s, int a, int na, int b, int nb, unsigned *out, int o, int d0,
                                           int d1) {
  if (d0 >= d1) return;
  int lo = max(0, d0 - nb), hi = min(d0, na);
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (s[padded(a + mid)] < s[padded(b + d0 - 1 - mid)]) lo = mid + 1;
    else hi = mid;
  }
  int i = a + lo, j = b + d0 - lo;
  const int ie = a + na, je = b + nb;
  unsigned x = i < ie ? s[padded(i)] : 0xffffffffu, y = j < je ? s[padded(j)] : 0xffffffffu;
  for (int d = d0; d < d1; d++) {
    const bool second = j < je && (i >= ie || y < x);
    out[padded(o + d)] = second ? y : x;
    const int next = second ? ++j : ++i;
    const unsigned v = next < (second ? je : ie) ? s[padded(next)] : 0xffffffffu;
    if (second) y = v;
    else x = v;
  }
}

// The words of keys[0, n), n <= kWarpSortCap, positions from `first` on, sorted by one warp; the result
// is in s or t (returned), padded positions from `first` on.
__device__ __forceinline__ unsigned *warp_sort_words(const unsigned long long *keys, unsigned *s, unsigned *t,
                                                     const WordForm &f, int first, int n) {
  const int n0 = min(n, kRunCap), n1 = n - n0;
  sort_run(keys, s, f, first, n0);
  if (n1 > 0) sort_run(keys + n0, s, f, first + n0, n1);
  __syncwarp();
  if (n1 <= 0) return s;
  const int lane = threadIdx.x & 31, part = (n + 31) >> 5;
  merge_part(s, first, n0, first + n0, n1, t, first, min(lane * part, n), min(lane * part + part, n));
  __syncwarp();
  return t;
}

// A segment of n <= kWarpSortCap keys, sorted by one warp. False: it needs all key bits.
__device__ __forceinline__ bool warp_sort_segment(const Work &w, const unsigned long long *keys, unsigned *sk, bool bnd,
                                                  long long s0, int n, int lane) {
  const WordForm f = word_form(key_range(keys, n, lane, 32), bnd, n);
  if (!f.ok) return false;
  unsigned *s = warp_sort_words(keys, sk, sk + kWarpWords, f, 0, n);
  if (!f.exact) {
    int pass = 0;
    while (__any_sync(0xffffffffu, exchange_ties(keys, s, Padded(), n, f.up, lane, 32, [] { __syncwarp(); })))
      if (++pass == kFixPasses) return false;
  }
  for (int i = lane; i < n; i += 32) store_sorted(w, bnd, s0 + i, word_key(f, keys, s[padded(i)]));
  __syncwarp();
  return true;
}

// Warps take groups of `grab` segments from a queue (tiles' Gaussian lists,
// then boundary lists), the lanes reading their bounds together, and sort the
// ones of up to kWarpSortCap keys: up to two runs in registers, a power-of-two
// number of words per lane, and a merge; longer ones, and those that need all
// key bits, are listed for k_tile_sort_big. Bound: instruction fetch and issue.
// One warp's radix sort of a segment in shared memory (four or five passes,
// each ranking 32 keys per round by a match) took 118 us on one 800^2 view
// and 0.77 ms on 64 mixed views (30 M keys); this network on 64-bit keys 25 us
// and 1.05 ms (its code did not stay in the instruction cache), on 32-bit
// words with up to 32 per lane 21 us and 0.58 ms, with the runs of 16 per lane
// and the merge 20 us and 0.48 ms.
__global__ void __launch_bounds__(kSortThreads, 6) k_tile_sort(Params p, Work w, int *big_list, int grab) {
  chained();
  __shared__ unsigned s_sort[2 * kSortWarps * kWarpWords];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const bool g_over = w.g_tstart[p.tiles] > p.max_pairs, b_over = w.b_tstart[p.tiles] > p.max_bpairs;
  const int items = 2 * p.tiles;
  unsigned *sk = s_sort + 2 * wp * kWarpWords;
  for (;;) {
    int base = 0;
    if (lane == 0) base = atomicAdd(w.counters + kQueueSort, grab);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (base >= items) break;
    bool bnd = false;
    long long s0 = 0, s1 = 0;
    const int item = base + lane;
    if (lane < grab && item < items) {
      segment_bounds(p, w, item, bnd, s0, s1);
      if (bnd ? b_over : g_over) s1 = s0;  // unwritten slots: nothing to sort
    }
    const int n_lane = (int)(s1 - s0);
    // the tile into its class's list (a list that overflowed counts as empty)
    const int cls = lane < grab && item < p.tiles ? (n_lane > 0) + (n_lane >= 128) + (n_lane >= 384) + (n_lane >= 768) : -1;
#pragma unroll
    for (int c = 0; c < kTileClasses; c++) {
      const unsigned m = __ballot_sync(0xffffffffu, cls == c);
      if (!m) continue;
      int at = 0;
      if (lane == 0) at = atomicAdd(w.counters + kTileClass + c, __popc(m));
      at = __shfl_sync(0xffffffffu, at, 0);
      if (cls == c) w.tile_order[(size_t)c * p.tiles + at + __popc(m & ((1u << lane) - 1u))] = item;
    }
    if (n_lane > kWarpSortCap) big_list[atomicAdd(w.counters + kBigCount, 1)] = item;
    unsigned todo = __ballot_sync(0xffffffffu, n_lane > 0 && n_lane <= kWarpSortCap);
    while (todo) {
      const int l = __ffs(todo) - 1;
      todo &= todo - 1;
      const int n = __shfl_sync(0xffffffffu, n_lane, l);
      const long long at = __shfl_sync(0xffffffffu, s0, l);
      const bool b = __shfl_sync(0xffffffffu, (int)bnd, l);
      const unsigned long long *keys = (b ? w.bkeys + p.max_bpairs : w.gkeys + p.max_pairs) + at;
      const bool ok = warp_sort_segment(w, keys, sk, b, at, n, lane);
      if (!ok && lane == 0) big_list[atomicAdd(w.counters + kBigCount, 1)] = (base + l) | kFullKeys;
      __syncwarp();
    }
  }
}

// keys of s[base, base + len) below `key` (with ties: not above it), len a power of two
template <class Key>
__device__ __forceinline__ int rank_in_run(const Key *s, int base, int len, Key key, bool ties) {
  int pos = 0;
  for (int step = len >> 1; step > 0; step >>= 1) {
    const Key v = s[padded(base + pos + step - 1)];
    if (ties ? v <= key : v < key) pos += step;
  }
  const Key v = s[padded(base + pos)];
  return pos + (int)(ties ? v <= key : v < key);
}

// 32 E keys of every warp of the block, in registers as loaded, sorted over
// the block into s (padded positions): each warp sorts its own in registers,
// then two merges (runs 0-1 and 2-3, then the two halves) in which each key,
// kept in its register, finds its rank in the other run by binary search and
// moves there. Equal keys (the padding) take the lower run's first, so that
// every position is written. Ends behind a block barrier.
template <int E, class Key>
__device__ __forceinline__ void block_sort(Key (&k)[E], Key *s) {
  constexpr int L = 32 * E;
  static_assert(kSortWarps == 4, "two merge levels");
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  warp_sort_regs<E>(k, lane);
  int pos[E];
#pragma unroll
  for (int e = 0; e < E; e++) {
    pos[e] = lane * E + e;
    s[padded(wp * L + pos[e])] = k[e];
  }
  for (int level = 0; level < 2; level++) {
    const int len = L << level, run = wp >> level;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; e++) pos[e] += rank_in_run(s, (run ^ 1) * len, len, k[e], run & 1);
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; e++) s[padded((run >> 1) * 2 * len + pos[e])] = k[e];
  }
  __syncthreads();
}

// a segment of n <= 128 E keys on all key bits
template <int E>
__device__ __forceinline__ void block_sort_full(const Work &w, const unsigned long long *keys, unsigned long long *s,
                                                bool bnd, long long s0, int n) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  unsigned long long k[E];
#pragma unroll
  for (int e = 0; e < E; e++) {
    const int i = wp * 32 * E + e * 32 + lane;
    k[e] = i < n ? keys[i] : ~0ull;
  }
  block_sort<E>(k, s);
  for (int i = threadIdx.x; i < n; i += kSortThreads) store_sorted(w, bnd, s0 + i, s[padded(i)]);
}

// the key range of a segment, by the block
__device__ __forceinline__ KeyRange block_key_range(const unsigned long long *keys, int n, KeyRange *s_range) {
  KeyRange r = key_range(keys, n, threadIdx.x, kSortThreads);
  if ((threadIdx.x & 31) == 0) s_range[threadIdx.x >> 5] = r;
  __syncthreads();
  for (int q = 0; q < kSortWarps; q++) {
    r.hi0 = min(r.hi0, s_range[q].hi0);
    r.hi1 = max(r.hi1, s_range[q].hi1);
    r.lo0 = min(r.lo0, s_range[q].lo0);
    r.lo1 = max(r.lo1, s_range[q].lo1);
  }
  return r;
}

// The words of keys[0, n), n <= kSortCap, positions from 0 on, sorted by the block: a quarter of them per
// warp, then two merges. s: both buffers; returned: the one that holds the result, behind a block barrier.
__device__ __forceinline__ unsigned *block_sort_run(const unsigned long long *keys, unsigned *s, const WordForm &f,
                                                    int n) {
  static_assert(kSortWarps == 4, "two merge levels");
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  unsigned *t = s + kSortWarps * kWarpWords;
  const int q = (n + kSortWarps - 1) / kSortWarps;  // <= kWarpSortCap, and all quarters on one side of kRunCap
  const int c[5] = {0, min(q, n), min(2 * q, n), min(3 * q, n), n};
  const int first = min(wp * q, n), mine = min(q, n - first);
  // one or two runs per warp: which buffer holds the result is decided by q for all warps alike
  sort_run(keys + first, s, f, first, min(mine, kRunCap));
  if (q > kRunCap) {
    const int n0 = min(mine, kRunCap), n1 = mine - n0, part = (mine + 31) >> 5;
    if (n1 > 0) sort_run(keys + first + n0, s, f, first + n0, n1);
    __syncwarp();
    merge_part(s, first, n0, first + n0, n1, t, first, min(lane * part, mine), min(lane * part + part, mine));
    unsigned *x = s; s = t; t = x;
  }
  __syncthreads();
  {  // quarters 0-1 by the first half of the block, 2-3 by the second
    const int h = wp >> 1, a = c[2 * h], b = c[2 * h + 1], e = c[2 * h + 2], part = (e - a + 63) >> 6;
    const int d = ((int)threadIdx.x & 63) * part;
    merge_part(s, a, b - a, b, e - b, t, a, min(d, e - a), min(d + part, e - a));
  }
  __syncthreads();
  {
    const int part = (n + kSortThreads - 1) / kSortThreads, d = (int)threadIdx.x * part;
    merge_part(t, 0, c[2], c[2], n - c[2], s, 0, min(d, n), min(d + part, n));
  }
  __syncthreads();
  return s;
}

// a segment of n <= kSortCap keys as 32-bit words; false: it needs all key bits
__device__ __forceinline__ bool block_sort_words(const Work &w, const unsigned long long *keys, unsigned *s,
                                                 KeyRange *s_range, bool bnd, long long s0, int n) {
  const WordForm f = word_form(block_key_range(keys, n, s_range), bnd, n);
  if (!f.ok) return false;
  s = block_sort_run(keys, s, f, n);
  if (!f.exact) {
    int pass = 0;
    while (__syncthreads_or(
        exchange_ties(keys, s, Padded(), n, f.up, threadIdx.x, kSortThreads, [] { __syncthreads(); })))
      if (++pass == kFixPasses) return false;
  }
  for (int i = threadIdx.x; i < n; i += kSortThreads)
    store_sorted(w, bnd, s0 + i, word_key(f, keys, s[padded(i)]));
  return true;
}

// How many of the first d outputs of the merge of a[0, na) and b[0, nb) (distinct words, global memory)
// come from a: the warp tests 32 points of the diagonal at a time.
__device__ __forceinline__ int merge_split(const unsigned *a, int na, const unsigned *b, int nb, int d) {
  const int lane = threadIdx.x & 31;
  int lo = max(0, d - nb), hi = min(d, na);
  while (lo < hi) {
    const int step = (hi - lo + 31) >> 5, mid = lo + lane * step;
    const bool below = mid < hi && a[mid] < b[d - 1 - mid];
    const int cnt = __popc(__ballot_sync(0xffffffffu, below));
    hi = min(hi, lo + cnt * step);
    if (cnt > 0) lo += (cnt - 1) * step + 1;
  }
  return lo;
}

// src[0, n) in sorted runs of len words merged in pairs into dst, kSortCap outputs at a time: their inputs
// are two contiguous pieces, merged in shared memory (s: both buffers).
__device__ __forceinline__ void merge_runs(const unsigned *src, unsigned *dst, int n, int len, unsigned *s, int *s_split) {
  unsigned *t = s + kSortWarps * kWarpWords;
  const int wp = threadIdx.x >> 5;
  for (int r = 0; r < n; r += 2 * len) {
    const int na = min(len, n - r), nb = min(len, n - r - na);
    const unsigned *a = src + r, *b = a + na;
    for (int d0 = 0; d0 < na + nb; d0 += kSortCap) {
      const int d1 = min(d0 + kSortCap, na + nb), m = d1 - d0;
      if (wp < 2) s_split[wp] = merge_split(a, na, b, nb, wp ? d1 : d0);
      __syncthreads();
      const int i0 = s_split[0], ni = s_split[1] - i0, j0 = d0 - i0;
      for (int k = threadIdx.x; k < m; k += kSortThreads) s[padded(k)] = k < ni ? a[i0 + k] : b[j0 + k - ni];
      __syncthreads();
      const int part = (m + kSortThreads - 1) / kSortThreads, d = (int)threadIdx.x * part;
      merge_part(s, 0, ni, ni, m - ni, t, 0, min(d, m), min(d + part, m));
      __syncthreads();
      for (int k = threadIdx.x; k < m; k += kSortThreads) dst[r + d0 + k] = t[padded(k)];
    }
  }
  __syncthreads();
}

// A segment of kSortCap < n <= kLongCap keys as 32-bit words: equal runs of at most kSortCap sorted in shared
// memory, the runs merged between the two halves of the list's own place (8 bytes per key hold two words
// per key), ending in the upper half. False: it needs all key bits.
__device__ __forceinline__ bool block_sort_long(const Work &w, const unsigned long long *keys, unsigned *s,
                                                KeyRange *s_range, int *s_split, bool bnd, long long s0, int n) {
  const WordForm f = word_form(block_key_range(keys, n, s_range), bnd, n);
  if (!f.ok) return false;
  const int runs = (n + kSortCap - 1) / kSortCap, len = (n + runs - 1) / runs;
  unsigned *lower = reinterpret_cast<unsigned *>((bnd ? w.bkeys : w.gkeys) + s0), *upper = lower + n;
  unsigned *cur = (32 - __clz(runs - 1)) & 1 ? lower : upper;  // an odd number of merge passes ends in the other half
  for (int r = 0; r < n; r += len) {
    const int m = min(len, n - r);
    const unsigned *out = block_sort_run(keys + r, s, f, m);
    for (int k = threadIdx.x; k < m; k += kSortThreads) cur[r + k] = out[padded(k)] + (f.exact ? 0u : (unsigned)r);
    __syncthreads();
  }
  for (int l = len; l < n; l *= 2) {
    unsigned *next = cur == lower ? upper : lower;
    merge_runs(cur, next, n, l, s, s_split);
    cur = next;
  }
  if (!f.exact) {
    int pass = 0;
    while (__syncthreads_or(exchange_ties(keys, upper, [](int i) { return i; }, n, f.up, threadIdx.x, kSortThreads,
                                          [] { __syncthreads(); })))
      if (++pass == kFixPasses) return false;
  }
  // keys [i, i + step) end at word 2 (i + step), at most n + i + step: no word is overwritten before it is read
  constexpr int kEach = 8, step = kEach * kSortThreads;
  for (int i = 0; i < n; i += step) {
    unsigned word[kEach];
#pragma unroll
    for (int e = 0; e < kEach; e++) {
      const int k = i + e * kSortThreads + (int)threadIdx.x;
      word[e] = k < n ? upper[k] : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < kEach; e++) {
      const int k = i + e * kSortThreads + (int)threadIdx.x;
      if (k < n) store_sorted(w, bnd, s0 + k, word_key(f, keys, word[e]));
    }
  }
  return true;
}

// Segments longer than kWarpSortCap and those that need all key bits: one
// block each, in shared memory up to kSortCap keys, as merged runs of that many
// up to kLongCap (from there on the words' depth bits, 32 less the position's, no
// longer tell neighbours apart), by a stable radix sort in global memory beyond and where the
// words do not resolve the order. On eight 1600 x 1200 views of a room
// a bitonic network of the block over 64-bit keys in shared memory took 1.62
// ms, quarters sorted by the warps and merged on 32-bit words 0.78 ms; with
// larger Gaussians (150 M pairs, lists up to ~9,000 keys) the radix sort
// of the lists beyond kSortCap (a pass per 8 key bits, three barriers per 128 keys) took
// the kernel to 9.9 ms, the merged runs to 5.2. All key bits are sorted in as few registers as the list
// fills: padded to kSortCap keys whatever its length, boundary lists of ~200 keys whose primitive and index
// ranges exceed 31 bits (320,000 primitives in random order) took the binning of eight views 18.2 ms, now 1.6.
__global__ void __launch_bounds__(kSortThreads, 4) k_tile_sort_big(Params p, Work w, const int *big_list) {
  chained();
  extern __shared__ __align__(16) unsigned long long s_keys[];
  __shared__ KeyRange s_range[kSortWarps];
  __shared__ int s_split[2];
  const int nbig = w.counters[kBigCount];
  for (int b = blockIdx.x; b < nbig; b += gridDim.x) {
    const int item = big_list[b];
    const bool full = item & kFullKeys;
    bool bnd;
    long long s0, s1;
    segment_bounds(p, w, item & ~kFullKeys, bnd, s0, s1);
    const int n = (int)(s1 - s0);
    unsigned long long *keys = (bnd ? w.bkeys + p.max_bpairs : w.gkeys + p.max_pairs) + s0;
    if (n <= kSortCap) {
      if (full || !block_sort_words(w, keys, reinterpret_cast<unsigned *>(s_keys), s_range, bnd, s0, n)) {
        __syncthreads();
        if (n <= 128) block_sort_full<1>(w, keys, s_keys, bnd, s0, n);
        else if (n <= 512) block_sort_full<4>(w, keys, s_keys, bnd, s0, n);
        else if (n <= 1024) block_sort_full<8>(w, keys, s_keys, bnd, s0, n);
        else if (n <= 2048) block_sort_full<16>(w, keys, s_keys, bnd, s0, n);
        else block_sort_full<kWarpSortCap / 32>(w, keys, s_keys, bnd, s0, n);
      }
    } else if (n > kLongCap ||
               !block_sort_long(w, keys, reinterpret_cast<unsigned *>(s_keys), s_range, s_split, bnd, s0, n)) {
      __syncthreads();
      unsigned long long *s_red = s_keys;  // 2 per warp
      int *s_hist = reinterpret_cast<int *>(s_keys + 2 * kSortWarps), *s_base = s_hist + 256;
      unsigned long long *out = (bnd ? w.bkeys : w.gkeys) + s0;
      radix_global(keys, out, n, s_hist, s_base, s_base + 256, s_red);
      if (bnd)
        for (int i = threadIdx.x; i < n; i += kSortThreads) store_sorted(w, true, s0 + i, out[i]);
    }
    __syncthreads();
  }
}

}  // namespace

int launch_scan_pair(int *in0, long long *out0, int *in1, long long *out1, int n, bool clear, bool overlap,
                     cudaStream_t st) {
  if (n <= kScanOne) chain_launch(overlap, k_scan_pair<1>, 1, kScanThreads, 0, st, in0, out0, in1, out1, n, clear);
  else chain_launch(overlap, k_scan_pair<kScanCluster>, kScanCluster, kScanThreads, 0, st, in0, out0, in1, out1, n, clear);
  return 1;
}

cudaError_t configure_binning() {
  return cudaFuncSetAttribute(k_tile_sort_big, cudaFuncAttributeMaxDynamicSharedMemorySize, kSortBigSmem);
}

int launch_binning(const Params &p, const Work &w, cudaStream_t st) {
  if (p.tiles <= 0) return 0;
  if (p.tiles <= kScanOne) chain_launch(p.P <= kOverlapPixels, k_tile_scan<1>, 1, kScanThreads, 0, st, p, w);
  else chain_launch(p.P <= kOverlapPixels, k_tile_scan<kScanCluster>, kScanCluster, kScanThreads, 0, st, p, w);
  chain_launch(p.P <= kOverlapPixels, k_emit, 16 * 152, 256, 0, st, p, w);
  // segments per dequeue: enough dequeues for every resident warp to take a few, so that long segments
  // spread, and few enough that the queue's one counter is no bottleneck
  const int blocks = 6 * 152, grab = std::max(1, std::min(32, 2 * p.tiles / (blocks * kSortWarps * 4)));
  chain_launch(p.P <= kOverlapPixels, k_tile_sort, blocks, kSortThreads, 0, st, p, w, w.big_list, grab);
  chain_launch(p.P <= kOverlapPixels, k_tile_sort_big, 4 * 152, kSortThreads, kSortBigSmem, st, p, w, w.big_list);
  return 4;
}

}  // namespace bgt
