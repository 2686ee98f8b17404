// Sub-primitive generation (Sec. 3.2, "Sub-Primitive Generation") and the
// boundary points of discontinuity-aware blending (same section, first
// paragraph of "Discontinuity-Aware Alpha Blending").
//
// For every foreground pixel q (I_id(q) = g >= 0) one Gaussian is placed at
// S_q = S(I_uv(q)) of primitive g (Eq. 3) with colour c_q (Eq. 4), the
// primitive's rotation / scale (Eq. 5 at attribute-map resolution 1) and the
// primitive's opacity; it is projected with the EWA approximation (J W
// Sigma3D W^T J^T + dilation) as in 3DGS. Pixels of B (a 4-neighbour with a
// different id) also yield a boundary point b = projection of the same S_q
// with radius sigma = k_b fx r_b / z.
//
// Gaussians and boundary points are compacted in global pixel order: k_ids
// turns the depth keys into I_id, finds B and counts both per block of pixels,
// its last block to finish scanning the counts; k_compact writes the
// foreground pixels (pixel, view, boundary index) at their ranks from the
// pixel bit masks of k_ids; the generation pass runs one thread per Gaussian,
// starting with the pixel's I_uv. Indices do not depend on scheduling. Each
// record counts its screen tiles into per-tile counters for the binning pass.
//
// I_uv is computed in the generation pass, where every lane holds a foreground
// pixel, not in a pass over all pixels whose background lanes idle; background
// pixels cost their depth key and their I_id only. The masks (1/4 byte per
// pixel) carry the counting pass's result to the compaction, which reads
// nothing else of a background pixel. Passes of their own for I_id and I_uv,
// the counts, their two scans, the totals and the compaction (eleven launches
// more) took 1.20 ms with the generation on 64 views of 256..1024 px squared
// (32 M pixels, 8.8 M Gaussians), 2.77 ms on eight 1600 x 1200 views of the
// room (15 M Gaussians) and 82 us on one 800^2 view; now 0.92 ms (k_ids 0.18,
// k_compact 0.05, k_generate 0.68), 1.6 ms and 44 us.
#include <algorithm>

#include "bgt_internal.cuh"

namespace bgt {

namespace {

constexpr int kGenThreads = 256;
constexpr int kGenWarps = kGenThreads / 32;
constexpr int kIdRounds = 8;                        // pixels per lane
constexpr int kChunk = 32 * kIdRounds;              // pixels of a warp
constexpr int kIdWords = kIdRounds * kGenWarps;     // mask words of a block
static_assert(kIdPixels == kChunk * kGenWarps && kIdWords == 64, "a warp scans a block's words two per lane");

// A warp chunk of kChunk pixels from `first`: its view when the whole chunk
// lies in one view (the usual case: one search and one division per chunk),
// with the view's size and the column and row of `first`; view = -1 otherwise.
struct ChunkPos {
  int view, W, H, x0, y0;
};

__device__ inline ChunkPos chunk_pos(const Params &p, const Work &w, int first) {
  ChunkPos c{-1, 1, 1, 0, 0};
  if (first >= p.P) return c;
  const int v = find_view(w.view_pix_off, p.V, first);
  if (min(first + kChunk, p.P) > __ldg(w.view_pix_off + v + 1)) return c;
  c.view = v;
  c.W = __ldg(&w.views[v].W);
  c.H = __ldg(&w.views[v].H);
  const int local = first - __ldg(w.view_pix_off + v);
  c.y0 = local / c.W;
  c.x0 = local - c.y0 * c.W;
  return c;
}

// I_id of a pixel from its depth key's low word (the winning flat triangle's id), -1 background
__device__ __forceinline__ int id_of(const Params &p, unsigned gid) {
  return gid == 0xffffffffu ? -1 : (int)prim_of(gid, p.nsub_inv);
}

__device__ __forceinline__ unsigned low_word(const unsigned long long *zbuf, int pix) {
  return reinterpret_cast<const unsigned *>(zbuf)[2 * (size_t)pix];
}

// Sigma3D of primitive m, whose rotation / scaling maps hold one texel (leg
// resolution 1), shared by its Gaussians
__device__ inline void prim_cov(const Scene &s, const Work &w, int m) {
  float qa[4], ls[3], Rm[9], sc3[3], S3[6];
#pragma unroll
  for (int k = 0; k < 4; k++) qa[k] = s.quat[4 * (size_t)m + k];
#pragma unroll
  for (int k = 0; k < 3; k++) ls[k] = s.log_scale[3 * (size_t)m + k];
  cov3d_f32(qa, ls, S3, Rm, sc3);
#pragma unroll
  for (int k = 0; k < 6; k++) w.prim_cov[6 * (size_t)m + k] = S3[k];
}

// I_id of every pixel, the foreground and boundary (4-neighbour of another id)
// bits of 32 pixels per word and their counts per block of kIdPixels pixels;
// the last block to finish scans the counts and stores F and Nb. The same
// launch clears the tile counters and the queue heads of the passes behind it
// and takes the primitives' Sigma3D, so that none of them is a launch. Bound:
// HBM (8 B read and 4 B written per pixel) and the loads' latency; loading every pixel's
// or every foreground pixel's rows above and below ahead of all rounds costs more
// registers than it hides (64 mixed views: 0.24 and 0.21 ms against 0.18).
__global__ void __launch_bounds__(kGenThreads) k_ids(Params p, Scene s, Work w, int npb) {
  chained();
  __shared__ int s_cnt[kGenWarps];  // foreground | boundary << 16
  __shared__ int2 s_sum[kGenWarps];
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gtid = blockIdx.x * kGenThreads + threadIdx.x, gthreads = gridDim.x * kGenThreads;
  for (int t = gtid; t < p.tiles; t += gthreads) {
    w.g_tcount[t] = 0;
    w.b_tcount[t] = 0;
    w.g_tfill[t] = 0;
    w.b_tfill[t] = 0;
  }
  if (gtid >= kQueueFwd && gtid < kCounters && gtid != kIdsDone) w.counters[gtid] = 0;
  if (p.attr_res == 1)
    for (int m = gtid; m < p.M; m += gthreads) prim_cov(s, w, m);
  if (blockIdx.x < npb) {
    const int first = blockIdx.x * kIdPixels + warp * kChunk;
    const ChunkPos cp = chunk_pos(p, w, first);
    int cnt = 0;
    unsigned gid[kIdRounds];
#pragma unroll
    for (int r = 0; r < kIdRounds; r++) {
      const int pix = first + r * 32 + lane;
      gid[r] = pix < p.P ? low_word(w.zbuf, pix) : 0xffffffffu;
    }
#pragma unroll
    for (int r = 0; r < kIdRounds; r++) {
      const int pix = first + r * 32 + lane;
      int id = id_of(p, gid[r]);
      if (id >= p.M) {
        atomicOr(w.status, kStatusBadPrim);
        id = -1;
      }
      const bool fg = id >= 0;
      const unsigned mf = __ballot_sync(0xffffffffu, fg);
      unsigned mb = 0u;
      if (mf) {
        int x = 0, y = 0, W = 1, H = 1;
        if (cp.view >= 0) {
          W = cp.W;
          H = cp.H;
          x = cp.x0 + r * 32 + lane;
          y = cp.y0;
          if (x >= W) {  // the chunk wraps to the following row(s)
            y += x / W;
            x -= (x / W) * W;
          }
        } else if (pix < p.P) {
          const int view = find_view(w.view_pix_off, p.V, pix);
          W = __ldg(&w.views[view].W);
          H = __ldg(&w.views[view].H);
          const int local = pix - __ldg(w.view_pix_off + view);
          y = local / W;
          x = local - y * W;
        }
        // a row's neighbours from the lanes beside, those of the warp's ends
        // and of the rows above and below from memory
        int il = __shfl_up_sync(0xffffffffu, id, 1), ir = __shfl_down_sync(0xffffffffu, id, 1);
        int iu = id, idn = id;
        if (fg) {
          if (x == 0) il = id;
          else if (lane == 0) il = id_of(p, low_word(w.zbuf, pix - 1));
          if (x == W - 1) ir = id;
          else if (lane == 31) ir = id_of(p, low_word(w.zbuf, pix + 1));
          if (y > 0) iu = id_of(p, low_word(w.zbuf, pix - W));
          if (y < H - 1) idn = id_of(p, low_word(w.zbuf, pix + W));
        }
        mb = __ballot_sync(0xffffffffu, fg && (il != id || ir != id || iu != id || idn != id));
      }
      if (pix < p.P) w.pid[pix] = id;
      if (lane == r) w.pix_mask[blockIdx.x * kIdWords + warp * kIdRounds + r] = make_uint2(mf, mb);
      cnt += __popc(mf) | (__popc(mb) << 16);
    }
    if (lane == 0) s_cnt[warp] = cnt;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (blockIdx.x < npb) {
      int2 t = make_int2(0, 0);
      for (int k = 0; k < kGenWarps; k++) {
        t.x += s_cnt[k] & 0xffff;
        t.y += s_cnt[k] >> 16;
      }
      w.blk_off[blockIdx.x] = t;
    }
    __threadfence();
    s_last = atomicAdd(w.counters + kIdsDone, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  // exclusive scan of the npb block counts, a run of consecutive blocks per thread
  __threadfence();
  const int per = (npb + kGenThreads - 1) / kGenThreads;
  const int b0 = min((int)threadIdx.x * per, npb), b1 = min(b0 + per, npb);
  int2 run = make_int2(0, 0);
  for (int b = b0; b < b1; b++) {
    const int2 c = __ldcg(w.blk_off + b);
    run.x += c.x;
    run.y += c.y;
  }
  int2 inc = run;
  for (int o = 1; o < 32; o <<= 1) {
    const int ax = __shfl_up_sync(0xffffffffu, inc.x, o), ay = __shfl_up_sync(0xffffffffu, inc.y, o);
    if (lane >= o) {
      inc.x += ax;
      inc.y += ay;
    }
  }
  if (lane == 31) s_sum[warp] = inc;
  __syncthreads();
  int2 off = make_int2(inc.x - run.x, inc.y - run.y);
  for (int k = 0; k < warp; k++) {
    off.x += s_sum[k].x;
    off.y += s_sum[k].y;
  }
  for (int b = b0; b < b1; b++) {
    const int2 c = __ldcg(w.blk_off + b);
    w.blk_off[b] = off;
    off.x += c.x;
    off.y += c.y;
  }
  if (threadIdx.x == kGenThreads - 1) {
    w.counters[kF] = off.x;
    w.counters[kNb] = off.y;
    w.counters[kIdsDone] = 0;
  }
}

// One count per tile of each lane's tile rect (x0 | y0 << 16, x1 | y1 << 16; empty when x0 > x1; `on`:
// the lane holds one). All lanes of the warp call it. Consecutive Gaussians are consecutive pixels, so
// their rects overlap: those of one view are counted over the tiles of their common bounding rect, one
// ballot per tile, lane t keeping the t-th tile's count, so that a warp issues one atomic instruction
// per 32 tiles. A match per lane and tile instead, each peer group adding with an atomic of its own,
// cost ~40 instructions per tile of the longest rect: on eight 1600 x 1200 views of the room (15 M
// Gaussians of ~3 tiles, 2 M boundary points) the generation pass took 3.7 ms, with the common rect 1.5
// ms. Rects far apart (a common rect of more than kRectSpan tiles: a warp whose pixels wrap to the next
// row of a wide object) are counted one tile at a time.
constexpr unsigned kRectSpan = 96;

__device__ __forceinline__ void count_tiles(int *cnt, bool on, int view, int tile_off, int tiles_x, uint2 rect) {
  const unsigned lane = threadIdx.x & 31;
  const unsigned x0 = rect.x & 0xffffu, y0 = rect.x >> 16, x1 = rect.y & 0xffffu, y1 = rect.y >> 16;
  on = on && x0 <= x1;
  unsigned todo = __ballot_sync(0xffffffffu, on);
  while (todo) {
    const int lead = __ffs(todo) - 1;
    const int lead_view = __shfl_sync(0xffffffffu, view, lead);  // by every lane, so not behind `on &&`
    const bool in = on && view == lead_view;
    todo &= ~__ballot_sync(0xffffffffu, in);
    const unsigned ux0 = __reduce_min_sync(0xffffffffu, in ? x0 : 0xffffu);
    const unsigned uy0 = __reduce_min_sync(0xffffffffu, in ? y0 : 0xffffu);
    const unsigned ux1 = __reduce_max_sync(0xffffffffu, in ? x1 : 0u);
    const unsigned uy1 = __reduce_max_sync(0xffffffffu, in ? y1 : 0u);
    const unsigned uw = ux1 - ux0 + 1u, area = uw * (uy1 - uy0 + 1u);
    if (area > kRectSpan) {
      if (in)
        for (unsigned y = y0; y <= y1; y++)
          for (unsigned x = x0; x <= x1; x++) atomicAdd(cnt + tile_off + y * (unsigned)tiles_x + x, 1);
      __syncwarp();
      continue;
    }
    const int off = __shfl_sync(0xffffffffu, tile_off, lead);
    const unsigned width = (unsigned)__shfl_sync(0xffffffffu, tiles_x, lead);
    unsigned x = ux0, y = uy0;
    for (unsigned t0 = 0; t0 < area; t0 += 32) {
      const unsigned n = min(area - t0, 32u);
      unsigned mine = 0u;
      for (unsigned t = 0; t < n; t++) {
        const unsigned m = __ballot_sync(0xffffffffu, in && x - x0 <= x1 - x0 && y - y0 <= y1 - y0);
        if (lane == t) mine = m;
        if (++x > ux1) {
          x = ux0;
          y++;
        }
      }
      const unsigned ay = (t0 + lane) / uw, ax = t0 + lane - ay * uw;
      if (mine) atomicAdd(cnt + off + (uy0 + ay) * width + ux0 + ax, __popc(mine));
    }
  }
}

// tile rect of the pixel box [cx - rx, cx + rx] x [cy - ry, cy + ry]; empty -> x0 > x1
__device__ inline uint2 tile_rect(float cx, float cy, float rx, float ry, const View &vw, int t) {
  int x0 = (int)ceilf(cx - rx), x1 = (int)floorf(cx + rx);
  int y0 = (int)ceilf(cy - ry), y1 = (int)floorf(cy + ry);
  x0 = max(x0, 0); y0 = max(y0, 0);
  x1 = min(x1, vw.W - 1); y1 = min(y1, vw.H - 1);
  if (x0 > x1 || y0 > y1) return make_uint2(1u, 0u);  // x0 = 1 > x1 = 0: empty
  const int sh = 31 - __clz(t);  // 8, 16 or 32; no coordinate is negative here
  x0 >>= sh; x1 >>= sh; y0 >>= sh; y1 >>= sh;
  return make_uint2((unsigned)x0 | ((unsigned)y0 << 16), (unsigned)x1 | ((unsigned)y1 << 16));
}

// compaction: each warp writes its chunk's foreground pixels at their ranks in
// pixel order (the Gaussian and boundary indices): the block's offset plus
// the set bits of the block's mask words before the pixel
__global__ void __launch_bounds__(kGenThreads) k_compact(Params p, Work w) {
  chained();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint2 *words = w.pix_mask + blockIdx.x * kIdWords;
  const uint2 m0 = words[lane], m1 = words[32 + lane];
  const uint2 mine = warp < kGenWarps / 2 ? m0 : m1;  // the half of the words holding this warp's
  const int w0 = (warp * kIdRounds) & 31;
  if (!__any_sync(0xffffffffu, lane >= w0 && lane < w0 + kIdRounds && mine.x)) return;
  const int c0 = __popc(m0.x) | (__popc(m0.y) << 16), c1 = __popc(m1.x) | (__popc(m1.y) << 16);
  int excl = warp < kGenWarps / 2 ? c0 : c1;
  const int own = excl;
  for (int o = 1; o < 32; o <<= 1) {
    const int a = __shfl_up_sync(0xffffffffu, excl, o);
    if (lane >= o) excl += a;
  }
  excl -= own;
  if (warp >= kGenWarps / 2) {
    int t = c0;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    excl += t;
  }
  const int2 off = w.blk_off[blockIdx.x];
  const int first = blockIdx.x * kIdPixels + warp * kChunk;
  const ChunkPos cp = chunk_pos(p, w, first);
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int r = 0; r < kIdRounds; r++) {
    const unsigned mf = __shfl_sync(0xffffffffu, mine.x, w0 + r), mb = __shfl_sync(0xffffffffu, mine.y, w0 + r);
    const int before = __shfl_sync(0xffffffffu, excl, w0 + r);
    if (!((mf >> lane) & 1u)) continue;
    const int pix = first + r * 32 + lane;
    const int gi = off.x + (before & 0xffff) + __popc(mf & lt);
    w.g_pix[gi] = pix;
    w.g_view[gi] = cp.view >= 0 ? cp.view : find_view(w.view_pix_off, p.V, pix);
    w.g_bidx[gi] = (mb >> lane) & 1u ? off.y + (before >> 16) + __popc(mb & lt) : -1;
    w.g_prim[gi] = w.pid[pix];
  }
}

// I_uv of pixel (qx, qy) from the winning flat triangle `sid` of the lattice of
// the primitive with control points cp: its three vertices by the raster's
// operations (weights tabulated in sB), then perspective-correct barycentrics
template <int N>
__device__ inline float2 pixel_uv(const float *sB, const float *cp, int sid, int L, const View &vw, float near_z,
                                  int qx, int qy) {
  constexpr int NCP = (N + 1) * (N + 2) / 2;
  float c[3 * NCP];
#pragma unroll
  for (int k = 0; k < 3 * NCP; k++) c[k] = __ldg(cp + k);
  int va[3], vb[3];
  subtri_verts(L, sid, va, vb);
  RVert r[3];
#pragma unroll
  for (int k = 0; k < 3; k++) r[k] = vertex_from_weights<N>(sB + vslot(va[k], vb[k], L) * NCP, c, vw, near_z);
  long long area2 = edge_fn(r[0].X, r[0].Y, r[1].X, r[1].Y, r[2].X, r[2].Y);
  if (area2 < 0) {
    RVert t = r[1]; r[1] = r[2]; r[2] = t;
    int x = va[1]; va[1] = va[2]; va[2] = x;
    x = vb[1]; vb[1] = vb[2]; vb[2] = x;
    area2 = -area2;
  }
  const int Px = qx * 256, Py = qy * 256;
  const long long e0 = edge_fn(r[1].X, r[1].Y, r[2].X, r[2].Y, Px, Py);
  const long long e1 = edge_fn(r[2].X, r[2].Y, r[0].X, r[0].Y, Px, Py);
  const long long e2 = edge_fn(r[0].X, r[0].Y, r[1].X, r[1].Y, Px, Py);
  const float af = (float)area2;
  const float w0 = ((float)e0 / af) / r[0].Z;
  const float w1 = ((float)e1 / af) / r[1].Z;
  const float w2 = ((float)e2 / af) / r[2].Z;
  const float ws = (w0 + w1) + w2;
  return make_float2((w0 * (float)va[0] + w1 * (float)va[1] + w2 * (float)va[2]) / (ws * (float)L),
                     (w0 * (float)vb[0] + w1 * (float)vb[1] + w2 * (float)vb[2]) / (ws * (float)L));
}

// One thread per Gaussian (sub-primitive) and boundary point. Bound: issue (IEEE divisions of I_uv and
// of the vertices, double-float placement), so registers are traded for occupancy: 4 blocks per SM at
// degrees 1-3 against 3 took 0.68 against 0.73 ms (degree 2, 8.8 M Gaussians) and 0.184 against 0.199
// ms (degree 3, 1.9 M); 5 blocks spill (0.79 ms).
template <int N>
__global__ void __launch_bounds__(kGenThreads, N <= 3 ? 4 : 3) k_generate(Params p, Scene s, Work w) {
  __shared__ float sB[kMaxVerts * SurfPoint<N>::M];
  tabulate_lattice<N>(p.L, sB);
  __syncthreads();
  chained();
  const int F = w.counters[kF];
  for (int g0 = blockIdx.x * kGenThreads; g0 < F; g0 += gridDim.x * kGenThreads) {
    // lanes past the last Gaussian repeat it without storing (the tile counts are taken by whole warps)
    const bool live = g0 + (int)threadIdx.x < F;
    const int gi = live ? g0 + (int)threadIdx.x : F - 1;
    const int pix = w.g_pix[gi], view = w.g_view[gi], bi = w.g_bidx[gi], prim = w.g_prim[gi];
    const View &vw = w.views[view];
    const int local = pix - vw.pix_off;
    const int qy = local / vw.W, qx = local - qy * vw.W;
    const float *cp = s.ctrl + (size_t)prim * p.ncp * 3;
    const float2 uv = pixel_uv<N>(sB, cp, (int)(low_word(w.zbuf, pix) - (unsigned)prim * (unsigned)(2 * p.L * p.L)), p.L,
                                  vw, p.near_z, qx, qy);
    SurfPoint<N> sp;
    surface_point<N>(cp, uv.x, uv.y, vw, sp);
    const float2 off = project_offset(sp.t, vw, qx, qy);
    const float tx = sp.t[0].hi + sp.t[0].lo, ty = sp.t[1].hi + sp.t[1].lo, tz = sp.t[2].hi + sp.t[2].lo;
    // depth sort key refinement: the exact depth hi + lo lies in the rounding
    // interval of tz; its position there, in 1/32 ulp, extends the FP32 bits
    // by 5 monotone bits (|lo| <= ulp / 2 maps to 0..31)
    unsigned char dsub = 16;
    {
      const df z = df_fast_two_sum(sp.t[2].hi, sp.t[2].lo);
      const float r = __fsub_rn(z.hi, tz) + z.lo;  // exact depth minus tz
      const float ulp = __int_as_float(__float_as_int(tz) & 0x7f800000) * 1.1920928955078125e-7f;
      if (ulp > 0.f) {
        const float c = floorf(r / ulp * 32.0f) + 16.0f;
        dsub = (unsigned char)fminf(fmaxf(c, 0.0f), 31.0f);
      }
    }
    // EWA: T = J W, Sigma2D = T Sigma3D T^T + dilation I
    const float iz = 1.0f / tz;
    const float j00 = vw.fx * iz, j02 = -vw.fx * tx * iz * iz;
    const float j11 = vw.fy * iz, j12 = -vw.fy * ty * iz * iz;
    float T0[3], T1[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
      T0[k] = j00 * vw.R[k] + j02 * vw.R[6 + k];
      T1[k] = j11 * vw.R[3 + k] + j12 * vw.R[6 + k];
    }
    // Sigma3D from the attribute maps interpolated at I_uv (Eq. 5); maps of leg
    // resolution 1 hold one texel, so Sigma3D is the primitive's
    float S3[6];
    if (p.attr_res == 1) {
#pragma unroll
      for (int k = 0; k < 6; k++) S3[k] = w.prim_cov[6 * (size_t)prim + k];
    } else {
      float qa[4], ls[3], Rm[9], sc3[3], tw[3];
      int tex[3];
      gauss_attrs(s.quat, s.log_scale, p.attr_res, p.ntex, prim, uv.x, uv.y, qa, ls, tex, tw);
      cov3d_f32(qa, ls, S3, Rm, sc3);
    }
    const float Sxx = S3[0], Sxy = S3[1], Sxz = S3[2], Syy = S3[3], Syz = S3[4], Szz = S3[5];
    const float a0 = T0[0] * Sxx + T0[1] * Sxy + T0[2] * Sxz;
    const float a1 = T0[0] * Sxy + T0[1] * Syy + T0[2] * Syz;
    const float a2 = T0[0] * Sxz + T0[1] * Syz + T0[2] * Szz;
    const float b0 = T1[0] * Sxx + T1[1] * Sxy + T1[2] * Sxz;
    const float b1 = T1[0] * Sxy + T1[1] * Syy + T1[2] * Syz;
    const float b2 = T1[0] * Sxz + T1[1] * Syz + T1[2] * Szz;
    const float cA = a0 * T0[0] + a1 * T0[1] + a2 * T0[2] + p.dilation;
    const float cB = a0 * T1[0] + a1 * T1[1] + a2 * T1[2];
    const float cC = b0 * T1[0] + b1 * T1[1] + b2 * T1[2] + p.dilation;
    const float det = cA * cC - cB * cB;
    const float idet = 1.0f / det;
    const float Ka = cC * idet, Kb = -cB * idet, Kc = cA * idet;
    float col[3] = {0.f, 0.f, 0.f};
    const float *cc = s.color + (size_t)prim * p.ncp * 3;
#pragma unroll
    for (int a = 0; a < SurfPoint<N>::M; a++) {
      col[0] = fmaf(sp.B[a], __ldg(cc + 3 * a + 0), col[0]);
      col[1] = fmaf(sp.B[a], __ldg(cc + 3 * a + 1), col[1]);
      col[2] = fmaf(sp.B[a], __ldg(cc + 3 * a + 2), col[2]);
    }
    const float o = __ldg(s.opacity + prim);
    const bool finite = isfinite(off.x) && isfinite(off.y) && isfinite(Ka) && isfinite(Kb) &&
                        isfinite(Kc) && det > 0.f && tz > 0.f;
    if (!finite) atomicOr(w.status, kStatusNonFinite);
    uint2 rect = make_uint2(1u, 0u);
    float rsup = -1.0f;
    if (finite && o > p.alpha_min) {
      // support {o G >= alpha_min} lies in the box |dx| <= sqrt(lvl Sigma_xx),
      // |dy| <= sqrt(lvl Sigma_yy), lvl = 2 ln(o / alpha_min); widened slightly
      const float lvl = 2.0f * (logf(o) - p.log_alpha_min);
      const float rx = sqrtf(lvl * cA) * 1.0001f + 1e-3f;
      const float ry = sqrtf(lvl * cC) * 1.0001f + 1e-3f;
      rsup = fmaxf(rx, ry);
      rect = tile_rect((float)qx + off.x, (float)qy + off.y, rx, ry, vw, p.tile);
    }
    count_tiles(w.g_tcount, live, view, vw.tile_off, vw.tiles_x, rect);
    const unsigned qxy = (unsigned)qx | ((unsigned)qy << 16);
    if (live) {
      w.gA[gi] = make_float4(off.x, off.y, __uint_as_float(qxy), rsup);
      w.gB[gi] = make_float4(Ka, Kb, Kc, o);
      w.gC[gi] = make_float4(col[0], col[1], col[2], __int_as_float(prim));
      w.g_uv[gi] = uv;
      w.g_depth[gi] = tz;
      w.g_rect[gi] = rect;
      w.g_dsub[gi] = dsub;
      float4 *ggz = reinterpret_cast<float4 *>(w.gg + 12 * (size_t)gi);
      ggz[0] = ggz[1] = ggz[2] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (!__any_sync(0xffffffffu, live && bi >= 0)) continue;
    // boundary point: the same surface point, radius sigma = k_b fx r_b / z
    const bool bnd = live && bi >= 0;
    const float sigma = p.k_b * vw.fx * __ldg(s.r_b + prim) / tz;
    uint2 brect = make_uint2(1u, 0u);
    if (finite && sigma > 0.f && isfinite(sigma)) {
      const float rr = sigma * 1.0001f + 1e-3f;
      brect = tile_rect((float)qx + off.x, (float)qy + off.y, rr, rr, vw, p.tile);
    }
    count_tiles(w.b_tcount, bnd, view, vw.tile_off, vw.tiles_x, brect);
    if (bnd) {
      w.bR[bi] = make_float4(__uint_as_float(qxy), off.x, off.y, 1.0f / sigma);
      w.b_pix[bi] = pix;
      w.b_prim[bi] = prim;
      w.b_view[bi] = view;
      w.b_uv[bi] = uv;
      w.b_sigma[bi] = sigma;
      w.b_z[bi] = tz;
      w.b_rect[bi] = brect;
      w.bg_grad[bi] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
}

}  // namespace

// View-dependent colour (SH bands 1..D of the primitive) added to the diffuse
// colour of every Gaussian, at the direction from the camera centre to S_q
// (R^T t in world coordinates, t the camera-space point of Eq. 3)
template <int N>
__global__ void __launch_bounds__(256) k_sh_color(Params p, Scene s, Work w) {
  chained();
  const int F = w.counters[kF];
  constexpr int m = SurfPoint<N>::M;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < F; i += gridDim.x * blockDim.x) {
    float4 C = w.gC[i];
    const int g = __float_as_int(C.w);
    const View &vw = w.views[w.g_view[i]];
    const float2 uv = w.g_uv[i];
    float B[m], S[3] = {0.f, 0.f, 0.f};
    bernstein_f32<N>(uv.x, uv.y, B);
    const float *cp = s.ctrl + (size_t)g * m * 3;
#pragma unroll
    for (int a = 0; a < m; a++)
#pragma unroll
      for (int c = 0; c < 3; c++) S[c] = fmaf(B[a], __ldg(cp + 3 * a + c), S[c]);
    float t[3], dv[3];
#pragma unroll
    for (int r = 0; r < 3; r++) t[r] = vw.R[3 * r] * S[0] + vw.R[3 * r + 1] * S[1] + vw.R[3 * r + 2] * S[2] + vw.t[r];
#pragma unroll
    for (int k = 0; k < 3; k++) dv[k] = vw.R[k] * t[0] + vw.R[3 + k] * t[1] + vw.R[6 + k] * t[2];
    const float inv = rsqrtf(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]);
    float Y[15];
    sh_eval(p.sh_deg, dv[0] * inv, dv[1] * inv, dv[2] * inv, Y);
    const float *shp = s.sh + (size_t)g * p.sh_k * 3;
#pragma unroll
    for (int k = 0; k < 15; k++) {
      if (k >= p.sh_k) break;
      C.x = fmaf(Y[k], __ldg(shp + 3 * k + 0), C.x);
      C.y = fmaf(Y[k], __ldg(shp + 3 * k + 1), C.y);
      C.z = fmaf(Y[k], __ldg(shp + 3 * k + 2), C.z);
    }
    w.gC[i] = C;
  }
}

// I_uv of every pixel from the Gaussians' (the background cleared before; Gaussians that were
// loaded for the binning stage on its own have no pixel of a raster)
__global__ void k_scatter_uv(Work w, int F, int P) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < F && (unsigned)w.g_pix[i] < (unsigned)P) w.puv[w.g_pix[i]] = w.g_uv[i];
}

void launch_scatter_uv(const Params &p, const Work &w, int F, cudaStream_t st) {
  cudaMemsetAsync(w.puv, 0, sizeof(float2) * (size_t)p.P, st);
  if (F > 0) k_scatter_uv<<<(F + 255) / 256, 256, 0, st>>>(w, F, p.P);
}

int launch_ids(const Params &p, const Scene &s, const Work &w, cudaStream_t st) {
  const int npb = (p.P + kIdPixels - 1) / kIdPixels;
  // small views of many primitives: more blocks for Sigma3D than the pixels give
  const int blocks = std::max(npb, std::min((p.M + kGenThreads - 1) / kGenThreads, num_sms()));
  chain_launch(p.P <= kOverlapPixels, k_ids, blocks, kGenThreads, 0, st, p, s, w, npb);
  return 1;
}

int launch_generate(const Params &p, const Scene &s, const Work &w, cudaStream_t st) {
  chain_launch(p.P <= kOverlapPixels, k_compact, (p.P + kIdPixels - 1) / kIdPixels, kGenThreads, 0, st, p, w);
  // one thread per Gaussian over a persistent grid (F is known on the device only)
  const int gblocks = std::min((p.P + kGenThreads - 1) / kGenThreads, num_sms() * 8);
  dispatch_degree(p.n, [&](auto d) { chain_launch(p.P <= kOverlapPixels, k_generate<decltype(d)::value>, gblocks, kGenThreads, 0, st, p, s, w); });
  int k = 2;
  if (p.sh_deg > 0) {
    dispatch_degree(p.n, [&](auto d) { chain_launch(p.P <= kOverlapPixels, k_sh_color<decltype(d)::value>, 152 * 8, 256, 0, st, p, s, w); });
    k++;
  }
  return k;
}

}  // namespace bgt
