// Photometric training loss of Sec. 3.3 (Eq. 9), L = (1 - lambda) L2 +
// lambda (1 - SSIM), and its gradient dL/dC with respect to the rendered
// image, in one fused kernel: the gradient lands in the layout the backward
// pass reads, and neither the windowed moments nor SSIM's partials ever
// leave shared memory.
//
// SSIM per channel: local moments under an 11 x 11 normalised Gaussian
// window (sigma 1.5, zero outside the image), C1 = 0.01^2, C2 = 0.03^2,
// averaged over pixels and channels; L2 is the mean of (C - C_gt)^2.
//
// One CTA owns a strip of kOutW columns (the first and the last of a view kR more)
// and some rows of one view, all three
// channels (views of any size, the image layout of the renderer: concatenated
// [H][W][3] blocks), and streams down it kRows rows at a time. The gradient
// needs SSIM's partials a = ds/dmu_x, b = ds/d(F (x^2 + y^2)), c = ds/d(F xy)
// on a 5-pixel halo, and those the image on a 10-pixel halo. Per group of
// rows: image values to a ring of rows in shared memory; the window along the
// rows over the four moments (x, y, x^2 + y^2, xy: SSIM needs the squares
// only in this sum); along the columns, one thread per column, into the sums
// of the eleven rows that a row reaches, which stay in registers from group to
// group; SSIM and its partials (zero at pixels outside the image, which are
// not in the mean) where a row's sums are complete; the window over the three
// partials the same way; gradient = 2 w_l2 (x - y) - w_ssim (F a + 2 x F b + y F
// c) with the symmetric window as its own adjoint. HBM traffic is the two
// images read and the gradient written.
//
// Streaming leaves a halo to recompute only beside a strip (64 of 54 columns, none beyond a
// view's edge) and above a segment of rows (none above the view): ~180 window FMAs per value, the square sum
// included, against 288 for 32 x 32 tiles that recompute it on all sides
// (52 x 52 -> 42 x 42 -> 32 x 32). Bound: issue (55 % of the slots busy at 12
// warps per SM) and the FP32 pipe. 64 mixed views (97 M values) took 2.01 ms,
// now 1.27; one 800^2 view 53 us, now 40; 64 and 112 views of 64^2 34 and 57 us while such a view took two
// strips and a search of 24 us, now 21 and 32 (tiles: 22 and 35). Views narrower than a strip leave the
// other columns idle: 112 views of 32^2 take 21 us, 13 as tiles. Three CTAs per SM spill the sums
// (112 registers: 1.70 ms without loads in flight, 2.13 with).
//
// The moments are taken of x - 1/2 and y - 1/2 (pixels outside the image: -1/2):
// variances and covariance do not move, and the cancellation in F x^2 -
// (F x)^2 loses two bits less. Error of the
// gradient against 64 bits on those views: 1.2e-5 of its norm, now 3.3e-6.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "bgt_internal.cuh"

namespace bgt {
namespace {

constexpr int kR = 5;
constexpr int kTaps = 2 * kR + 1;
constexpr int kLossThreads = 192;                       // 3 channels x 64 columns
constexpr int kOutW = 54, kPartW = kOutW + 2 * kR, kInW = kOutW + 4 * kR;  // columns: step of strips, partials, image
constexpr int kRows = 8;                                // rows per group
constexpr int kRun = 8;                                 // columns a thread filters along a row
constexpr int kRing = kRows + 2 * kR;                   // image rows held: an output row completes 10 rows behind
static_assert(kLossThreads == 3 * kPartW && kPartW == kRun * (kLossThreads / 3 / kRows), "one item per thread and phase");
// Shared-memory strides: one element of padding per 8, so that threads whose
// runs start 8 apart hit distinct banks; the ring's rows 16 banks apart (a half
// warp reads 8 runs of 2 rows), its channels 12 (three channels stored together)
__host__ __device__ constexpr int pad8(int i) { return i + (i >> 3); }
constexpr int kInStride = 88, kInPlane = kRing * kInStride + 6;  // float2 (x, y)
// rows of partials hold 8 columns of padding before and 5 behind, zero: the window along a row reads kR beyond
constexpr int kPartPad = 8, kPartAt = pad8(kPartPad);  // column c at pad8(c) + kPartAt
constexpr int kPartStride = pad8(kPartPad + kPartW + kR - 1) + 1, kPartPlane = kRows * kPartStride;  // float4
static_assert(pad8(kInW - 1) < kInStride && kInStride * 2 % 32 == 16, "ring row");
constexpr int kLossSmem = (int)(sizeof(float2) * 3 * kInPlane + sizeof(float4) * 3 * kPartPlane);
static_assert(2 * kLossSmem + 4096 <= 232448, "two CTAs per SM");
constexpr int kExtra = 3 * kInW - kLossThreads;         // values of an image row beyond one per thread
constexpr int kExtraLoads = (kExtra * kRows + kLossThreads - 1) / kLossThreads;
constexpr float kShift = 0.5f;

constexpr float kC1 = 0.01f * 0.01f;
constexpr float kC2 = 0.03f * 0.03f;

constexpr int kMaxLossViews = 112;  // views per launch: the table stays in 4 KB of parameters

// Two FP32 lanes in one 64-bit register: sm_100+ packed FMA / multiply, each
// lane rounded like fmaf / a single multiply.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ f32x2 pk(float2 v) { return pk(v.x, v.y); }
__device__ __forceinline__ float2 unpk(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

struct LossView {
  long long off;       // first pixel of the view in the concatenated images
  int W, H, strips, tile0;
  float w_l2, w_ssim;  // scale (1 - lambda) / N and scale lambda / N, N = 3 W H
};

struct LossArgs {
  const float *img, *gt;
  float *dimg, *loss;
  int n_views, seg;    // seg: output rows of a CTA
  float g[kTaps];      // 1-D window weights
  f32x2 g2[kTaps];     // the same, each weight in both lanes
  LossView view[kMaxLossViews];
};
static_assert(sizeof(LossArgs) <= 4000, "kernel parameters");

__global__ void __launch_bounds__(kLossThreads, 2) k_l2_dssim_grad(const __grid_constant__ LossArgs a) {
  chained();
  extern __shared__ float4 sm4[];
  float4 *part = sm4;                                             // [3][kRows][kPartStride] rows of moments / partials
  float2 *ring = reinterpret_cast<float2 *>(sm4 + 3 * kPartPlane);  // [3][kRing][kInStride] (x, y)
  __shared__ float s_red[kLossThreads / 32];

  // the view this CTA belongs to: last view whose first tile is <= blockIdx.x
  int lo = 0, hi = a.n_views - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.view[mid].tile0 <= (int)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const LossView &vw = a.view[lo];
  const int W = vw.W, H = vw.H;
  const int tile = blockIdx.x - vw.tile0;
  const int strip = tile % vw.strips;
  const int x0 = strip * kOutW, y0 = (tile / vw.strips) * a.seg;  // first column of partials, first output row
  const int y1 = min(y0 + a.seg, H);
  const int skip = max(2 * kR - y0, 0), r0 = y0 - 2 * kR + skip;  // rows above the view, first image row
  const float w_l2 = vw.w_l2, w_ssim = vw.w_ssim;
  const int tid = threadIdx.x;
  const int ch = tid / kPartW, col = tid % kPartW;    // column phases: channel and column
  const int hrow = col / (kPartW / kRun), hrun = col % (kPartW / kRun);  // row phases: row and run of columns
  float4 *pch = part + ch * kPartPlane;
  const float2 *rch = ring + ch * kInPlane;

  // loads: value e of an image row (pixel e / 3, channel e % 3) by thread e, the
  // kExtra values beyond one per thread spread over the threads
  // (plain loads: the renderer may still write the image when this kernel's blocks start, and the
  // read-only path of __ldg is for memory that nothing writes during the kernel)
  const long long pitch = 3ll * W;
  const long long origin = (vw.off + (long long)r0 * W + x0 - kR) * 3;  // of the first image row's values
  const int gx = x0 - kR + tid / 3;
  const bool col_ok = gx >= 0 && gx < W;
  const int slot_e = (tid % 3) * kInPlane + pad8(tid / 3);
  float2 ld[kRows], lx[kExtraLoads];
  auto load = [&](int i0) {  // image rows i0 .. i0 + kRows - 1 of the strip into registers
#pragma unroll
    for (int r = 0; r < kRows; r++) {
      ld[r] = make_float2(0.f, 0.f);
      if (col_ok && r0 + i0 + r < H) {
        const long long o = origin + (i0 + r) * pitch + tid;
        ld[r] = make_float2(a.img[o], a.gt[o]);
      }
    }
#pragma unroll
    for (int k = 0; k < kExtraLoads; k++) {
      const int q = tid + k * kLossThreads, r = q / kExtra, e = kLossThreads + q % kExtra;
      const int x = x0 - kR + e / 3;
      lx[k] = make_float2(0.f, 0.f);
      if (r < kRows && x >= 0 && x < W && r0 + i0 + r < H) {
        const long long o = origin + (i0 + r) * pitch + e;
        lx[k] = make_float2(a.img[o], a.gt[o]);
      }
    }
  };

  // sums of the rows begun: moments of rows i0 - 5 .. i0 + 4 (image rows of the strip), partials five rows behind
  f32x2 m01[2 * kR], m23[2 * kR], fab[2 * kR];
  float fc[2 * kR];
#pragma unroll
  for (int k = 0; k < 2 * kR; k++) {
    m01[k] = m23[k] = fab[k] = 0ull;
    fc[k] = 0.f;
  }
  if (skip > 0) {  // the rows above the view (x = y = 0), all of the same sums along the row
    const f32x2 xy2 = pk(-kShift, -kShift), sp = pk(2.f * kShift * kShift, kShift * kShift);
    f32x2 u = 0ull, v = 0ull;
#pragma unroll
    for (int t = 0; t < kTaps; t++) {
      u = fma2(a.g2[t], xy2, u);
      v = fma2(a.g2[t], sp, v);
    }
    for (int r = 0; r < skip; r++) {
#pragma unroll
      for (int k = 0; k + 1 < 2 * kR; k++) {
        m01[k] = fma2(a.g2[k + 1], u, m01[k + 1]);
        m23[k] = fma2(a.g2[k + 1], v, m23[k + 1]);
      }
      m01[2 * kR - 1] = mul2(a.g2[kTaps - 1], u);
      m23[2 * kR - 1] = mul2(a.g2[kTaps - 1], v);
    }
  }
  for (int k = tid; k < 3 * kRows * 2 * kR; k += kLossThreads) {  // the padding of the partials
    const int c = k % (2 * kR) < kR ? k % (2 * kR) - kR : k % (2 * kR) - kR + kPartW;
    part[k / (2 * kR) * kPartStride + pad8(c + kPartPad)] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float acc = 0.f;
  const int n_rows = y1 - r0 + 2 * kR;
  // output columns of the strip: at the view's edges the window's other half holds no partials
  const bool own = (strip == 0 || col >= kR) && (strip == vw.strips - 1 || col < kR + kOutW) && x0 + col < W;
  load(0);
  int base = 0;  // ring slot of image row i0
  for (int i0 = 0; i0 < n_rows; i0 += kRows) {
#pragma unroll
    for (int r = 0; r < kRows; r++) {
      int s = base + r;
      s -= s >= kRing ? kRing : 0;
      ring[slot_e + s * kInStride] = ld[r];
    }
#pragma unroll
    for (int k = 0; k < kExtraLoads; k++) {
      const int q = tid + k * kLossThreads, r = q / kExtra, e = kLossThreads + q % kExtra;
      int s = base + r;
      s -= s >= kRing ? kRing : 0;
      if (r < kRows) ring[(e % 3) * kInPlane + s * kInStride + pad8(e / 3)] = lx[k];
    }
    __syncthreads();
    if (i0 + kRows < n_rows) load(i0 + kRows);  // in flight over the phases below

    // along the rows: moments of kRun columns of one row
    {
      int s = base + hrow;
      s -= s >= kRing ? kRing : 0;
      const float2 *in = rch + s * kInStride + hrun * (kRun + 1);
      f32x2 h01[kRun], h23[kRun];
#pragma unroll
      for (int j = 0; j < kRun; j++) h01[j] = h23[j] = 0ull;
      const f32x2 shift = pk(-kShift, -kShift);
#pragma unroll
      for (int i = 0; i < kRun + 2 * kR; i++) {
        const f32x2 xy2 = add2(pk(in[i + (i >> 3)]), shift);
        const float2 v = unpk(xy2);
        const f32x2 sp = pk(fmaf(v.x, v.x, v.y * v.y), v.x * v.y);
#pragma unroll
        for (int j = 0; j < kRun; j++) {
          const int t = i - j;
          if (t >= 0 && t < kTaps) {
            h01[j] = fma2(a.g2[t], xy2, h01[j]);
            h23[j] = fma2(a.g2[t], sp, h23[j]);
          }
        }
      }
      float4 *o = pch + hrow * kPartStride + hrun * (kRun + 1) + kPartAt;
#pragma unroll
      for (int j = 0; j < kRun; j++) {
        const float2 u = unpk(h01[j]), v = unpk(h23[j]);
        o[j] = make_float4(u.x, u.y, v.x, v.y);
      }
    }
    __syncthreads();

    // along the columns: image row i0 + r completes the moments of row i0 + r - 5, in place
    {
      const bool x_ok = x0 + col < W;
      f32x2 s01[kRows + 2 * kR], s23[kRows + 2 * kR];
#pragma unroll
      for (int k = 0; k < 2 * kR; k++) {
        s01[k] = m01[k];
        s23[k] = m23[k];
      }
#pragma unroll
      for (int r = 0; r < kRows; r++) {
        float4 *cell = pch + r * kPartStride + pad8(col) + kPartAt;
        const float4 h = *cell;
        const f32x2 u = pk(h.x, h.y), v = pk(h.z, h.w);
#pragma unroll
        for (int t = 0; t < kTaps - 1; t++) {
          s01[r + t] = fma2(a.g2[t], u, s01[r + t]);
          s23[r + t] = fma2(a.g2[t], v, s23[r + t]);
        }
        s01[r + kTaps - 1] = mul2(a.g2[kTaps - 1], u);
        s23[r + kTaps - 1] = mul2(a.g2[kTaps - 1], v);
        const int gyp = r0 - kR + i0 + r;  // its row in the view
        float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
        if (x_ok && gyp >= 0 && gyp < H && gyp >= y0 - kR) {
          const float2 mu = unpk(s01[r]), sp = unpk(s23[r]);
          const float mx = mu.x + kShift, my = mu.y + kShift;
          const float l1 = 2.f * mx * my + kC1;
          const float cs1 = 2.f * (sp.y - mu.x * mu.y) + kC2;
          const float l2 = mx * mx + my * my + kC1;
          const float cs2 = (sp.x - (mu.x * mu.x + mu.y * mu.y)) + kC2;
          const float rD = __fdividef(1.f, l2 * cs2);  // D in [C1 C2, 4 (1 + C1) (2 + C2)]
          const float s = l1 * cs1 * rD;
          const float dN = 2.f * (my * cs1 - mu.y * l1);
          const float dD = 2.f * (mx * cs2 - mu.x * l2);
          d.x = (dN - s * dD) * rD;
          d.y = -s * l2 * rD;
          d.z = 2.f * l1 * rD;
          if (own && gyp >= y0 && gyp < y1) acc += w_ssim * (1.f - s);
        }
        *cell = d;
      }
#pragma unroll
      for (int k = 0; k < 2 * kR; k++) {
        m01[k] = s01[kRows + k];
        m23[k] = s23[kRows + k];
      }
    }
    __syncthreads();

    // along the rows of the partials (output columns that the strip does not own have a cut window)
    float4 h2[kRun];
    {
      const float4 *in = pch + hrow * kPartStride + hrun * (kRun + 1);  // column 8 hrun - 8
      constexpr int kLead = kPartPad - kR;
      f32x2 hab[kRun];
      float hc[kRun];
#pragma unroll
      for (int j = 0; j < kRun; j++) {
        hab[j] = 0ull;
        hc[j] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < kRun + 2 * kR; i++) {
        const float4 d = in[pad8(i + kLead)];
        const f32x2 u = pk(d.x, d.y);
#pragma unroll
        for (int j = 0; j < kRun; j++) {
          const int t = i - j;
          if (t >= 0 && t < kTaps) {
            hab[j] = fma2(a.g2[t], u, hab[j]);
            hc[j] = fmaf(a.g[t], d.z, hc[j]);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < kRun; j++) {
        const float2 u = unpk(hab[j]);
        h2[j] = make_float4(u.x, u.y, hc[j], 0.f);
      }
    }
    __syncthreads();
    {
      float4 *o = pch + hrow * kPartStride + hrun * (kRun + 1) + kPartAt;
#pragma unroll
      for (int j = 0; j < kRun; j++) o[j] = h2[j];
    }
    __syncthreads();

    // along the columns of the partials: image row i0 + r completes output row i0 + r - 10
    {
      f32x2 sab[kRows + 2 * kR];
      float sc[kRows + 2 * kR];
#pragma unroll
      for (int k = 0; k < 2 * kR; k++) {
        sab[k] = fab[k];
        sc[k] = fc[k];
      }
#pragma unroll
      for (int r = 0; r < kRows; r++) {
        const float4 h = pch[r * kPartStride + pad8(col) + kPartAt];
        const f32x2 u = pk(h.x, h.y);
#pragma unroll
        for (int t = 0; t < kTaps - 1; t++) {
          sab[r + t] = fma2(a.g2[t], u, sab[r + t]);
          sc[r + t] = fmaf(a.g[t], h.z, sc[r + t]);
        }
        sab[r + kTaps - 1] = mul2(a.g2[kTaps - 1], u);
        sc[r + kTaps - 1] = a.g[kTaps - 1] * h.z;
        const int gyo = r0 - 2 * kR + i0 + r;
        if (own && gyo >= y0 && gyo < y1) {
          int s = base + r - 2 * kR;  // the ring's oldest rows
          s += s < 0 ? kRing : 0;
          const float2 v = rch[s * kInStride + pad8(col + kR)];
          const float2 f = unpk(sab[r]);
          const float diff = v.x - v.y;
          const float dssim = f.x + 2.f * (v.x - kShift) * f.y + (v.y - kShift) * sc[r];
          a.dimg[(vw.off + (long long)gyo * W + x0 + col) * 3 + ch] = 2.f * w_l2 * diff - w_ssim * dssim;
          acc += w_l2 * diff * diff;
        }
      }
#pragma unroll
      for (int k = 0; k < 2 * kR; k++) {
        fab[k] = sab[kRows + k];
        fc[k] = sc[kRows + k];
      }
    }
    __syncthreads();
    base += kRows;
    base -= base >= kRing ? kRing : 0;
  }

  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((tid & 31) == 0) s_red[tid >> 5] = acc;
  __syncthreads();
  if (tid == 0 && a.loss) {
    float t = 0.f;
    for (int k = 0; k < kLossThreads / 32; ++k) t += s_red[k];
    atomicAdd(a.loss, t);
  }
}

// Output rows per CTA of a launch over views[0, n): the length whose waves of
// CTAs take the fewest groups of rows, the halo's 4 kR rows included (half of it in a view's first rows).
// One CTA per SM takes 3.4 us a group, two together 4.9, so a last wave that leaves half of the slots idle
// counts 7 of 10. Lengths are tried where the rows alone, without the rounding to segments and
// waves, could beat the best so far, and views of one height are counted
// together: 127 lengths over every view took 24 us at 64 views and 37 at 112, now 1 to 2 (5 at 112
// heights).
int loss_segment(const LossView *views, int n, int slots) {
  struct { unsigned H; long long strips; } of[kMaxLossViews];
  int m = 0;
  long long strips = 0, rows = 0;
  unsigned tall = 0;
  for (int v = 0; v < n; ++v) {
    const unsigned H = views[v].H;
    int k = m - 1;
    while (k >= 0 && k >= m - 8 && of[k].H != H) --k;
    if (k < 0 || k < m - 8) {
      k = m++;
      of[k].H = H;
      of[k].strips = 0;
    }
    of[k].strips += views[v].strips;
    strips += views[v].strips;
    rows += (long long)views[v].strips * H;
    tall = std::max(tall, H);
  }
  const auto cost = [&](unsigned seg, long long ctas) {
    const unsigned r = seg >= tall ? tall + 2 * kR : std::max(seg + 2 * kR, std::min(seg, tall - seg) + 4 * kR);
    const long long rem = ctas % slots;
    return (ctas / slots * 10 + (rem == 0 ? 0 : 2 * rem <= slots ? 7 : 10)) * ((r + kRows - 1) / kRows);
  };
  const auto bound = [&](unsigned seg) { return cost(seg, std::max(strips, (rows + seg - 1) / seg)); };
  const auto exact = [&](unsigned seg) {
    const unsigned long long inv = ((1ull << 32) + seg - 1) / seg;  // H / seg for H below 4 M, about beyond
    long long ctas = 0;
    for (int k = 0; k < m; ++k) ctas += of[k].strips * (long long)(((of[k].H - 1) * inv >> 32) + 1);
    return cost(seg, ctas);
  };
  constexpr unsigned kFirst = 4, kLast = 1020, kMid = 124;
  if (exact(kFirst) <= cost(kFirst, 1)) return (int)kFirst;  // one CTA per SM at most: no length has fewer groups
  const unsigned step = m <= 16 ? 4 : 16;  // the more heights, the less one length fits all of them
  const auto next = [&](unsigned seg) { return seg + (seg < kMid ? step : 2 * step); };
  long long bounds[(kMid - kFirst) / 4 + (kLast - kMid) / 8 + 2];
  unsigned best = kFirst;
  int q = 0, q_low = 0;
  for (unsigned seg = kFirst; seg <= kLast; seg = next(seg), ++q) {
    bounds[q] = bound(seg);
    if (bounds[q] < bounds[q_low]) {
      q_low = q;
      best = seg;
    }
  }
  long long best_cost = exact(best);
  q = 0;
  for (unsigned seg = kFirst; seg <= kLast; seg = next(seg), ++q) {
    if (bounds[q] >= best_cost) continue;
    const long long c = exact(seg);
    if (c < best_cost) {
      best_cost = c;
      best = seg;
    }
  }
  return (int)best;
}

}  // namespace

int launch_l2_dssim_grad(const float *img, const float *gt, int n_views, const int *sizes, float lambda,
                         float scale, float *dimg, float *loss, cudaStream_t st) {
  LossArgs a;
  a.img = img;
  a.gt = gt;
  a.dimg = dimg;
  a.loss = loss;
  double g[kTaps], sum = 0.0;
  for (int t = 0; t < kTaps; ++t) {
    const double d = t - kR;
    g[t] = std::exp(-d * d / (2.0 * 1.5 * 1.5));
    sum += g[t];
  }
  for (int t = 0; t < kTaps; ++t) {
    a.g[t] = (float)(g[t] / sum);
    unsigned int bits;
    std::memcpy(&bits, &a.g[t], sizeof(bits));
    a.g2[t] = ((unsigned long long)bits << 32) | bits;
  }
  cudaFuncSetAttribute(k_l2_dssim_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, kLossSmem);
  int launches = 0;
  long long off = 0;
  for (int v0 = 0; v0 < n_views; v0 += kMaxLossViews) {
    a.n_views = 0;
    for (int v = v0; v < n_views && v < v0 + kMaxLossViews; ++v) {
      const int W = sizes[2 * v], H = sizes[2 * v + 1];
      const long long npx = (long long)W * H;
      if (npx > 0) {
        LossView &r = a.view[a.n_views++];
        r.off = off;
        r.W = W;
        r.H = H;
        r.strips = std::max(1, (W - 2 * kR + kOutW - 1) / kOutW);  // the first and the last own kR columns more
        const double n = 3.0 * (double)npx;
        r.w_l2 = (float)((double)scale * (1.0 - (double)lambda) / n);
        r.w_ssim = (float)((double)scale * (double)lambda / n);
      }
      off += npx;
    }
    if (a.n_views == 0) continue;
    a.seg = loss_segment(a.view, a.n_views, 2 * num_sms());
    int tiles = 0;
    for (int v = 0; v < a.n_views; ++v) {
      LossView &r = a.view[v];
      r.tile0 = tiles;
      tiles += r.strips * ((r.H + a.seg - 1) / a.seg);
    }
    chain_launch(off <= kOverlapPixels, k_l2_dssim_grad, tiles, kLossThreads, kLossSmem, st, a);
    ++launches;
  }
  return launches;
}

}  // namespace bgt
