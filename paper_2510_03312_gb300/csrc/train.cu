// train.cu -- the training step around the rasterizer: the image loss of
// Sec. 4.5 with its gradient (ubs_image_loss) and the optimiser step of
// Sec. 5.1 fused with the activations, penalties and noise of Sec. 4.5
// (ubs_adam_step).
//
// Image loss, per view, L = (1 - lambda) L1 + lambda (1 - SSIM): L1 the mean
// |x - y| over pixels and channels, SSIM the mean map of Wang et al. (2004)
// per channel under an 11 x 11 Gaussian window (sigma 1.5), zero-padded.
// With the window statistics mu_x = G * x, E_xx = G * x^2, E_xy = G * (x y)
// (and the same for y), the map is
//   S = A B / (Cc D),  A = 2 mu_x mu_y + C1,  B = 2 (E_xy - mu_x mu_y) + C2,
//   Cc = mu_x^2 + mu_y^2 + C1,  D = (E_xx - mu_x^2) + (E_yy - mu_y^2) + C2,
// and its gradient with respect to x at pixel q gathers, over the output
// pixels p whose window covers q,
//   dS/dx(q) = sum_p G(p - q) [S_mu(p) + 2 x(q) S_xx(p) + y(q) S_xy(p)]
// with S_mu = dS/dmu_x (through A, B, Cc, D), S_xx = dS/dE_xx = dS/dD and
// S_xy = dS/dE_xy = 2 dS/dB.  G is symmetric and separable; both kernels take
// the rows first.  A CTA walks down a strip of kLT columns, a thread per
// column: every kLR rows are copied to shared memory with their halo
// (asynchronously, a step ahead), each thread sums the window along one row
// for four neighbouring columns, the warp exchanges those sums, and a row's
// sums enter the column's ten unfinished column sums, held in registers (sum i
// becomes sum i + 1 plus its tap: nothing is shifted or staged).  The strips'
// height is chosen so that all CTAs are resident at once, up to 96 rows.  Few or
// narrow images go by 32 x 32 tiles instead (use_tiles).
//   ssim_fwd_kernel   the five window statistics, S, the three partials (to
//                     the workspace) and per-block sums of S and |x - y|
//   ssim_bwd_kernel   the three partials convolved back, combined with the
//                     L1 term into dL/dimage; its first block reduces the
//                     block sums to the losses, in a fixed order
//                     (deterministic).
// Bound by instruction issue (2.8 of 4 a cycle forward; 60% of them the
// window's multiplies and adds) at 20 warps per SM.  1600 x 1060: 50 + 50 us
// and two reducing launches of 9 (32 x 32 tiles staged whole, both passes
// through shared memory: 45M + 36M warp instructions, 76% of the
// shared-memory pipe) -> 46 + 36 us (36M + 26M).  The order of every sum of a
// pixel is that of the row pass, then the column pass, from the first tap on.
//
// Adam (Kingma and Ba 2015) runs one thread per four parameters (16-byte loads
// and stores), reading raw, grad, m, v and writing raw, m, v and the activated
// value the rasterizer reads: 32 bytes of traffic per parameter.
#include <math.h>
#include <string.h>

#include "ubs.h"
#include "kernels.cuh"

namespace ubs {
namespace {

constexpr int kLossMaxViews = 256;
constexpr int kWin = 11, kRad = 5;
constexpr int kSumTile = 32;          // the workspace has a block sum per 32 x 32 pixels of a channel
constexpr int kLT = 128;              // threads: output columns of a strip
constexpr int kLW = kLT + 2 * kRad;   // its columns with the halo
constexpr int kLR = 4;                // rows per step
constexpr int kLossCtas = 5;          // CTAs per SM
constexpr uint64_t kMinRows = 32, kMaxRows = 96;  // height of a strip
constexpr float kC1 = 0.0001f, kC2 = 0.0009f;  // (0.01)^2, (0.03)^2

struct LossView {
  int32_t W, H, tiles_x;  // blocks (strips or tiles) across
  uint32_t pix_off;       // first pixel of the view
  uint32_t blk_off;       // first block of the view
  int32_t tiles;          // blocks per channel
};
struct LossParams {
  LossView v[kLossMaxViews];
  float2 g2[kRad + 1]; // 1-D window (g_k, g_k), g_k = g_(10 - k), sums to 1
  int32_t cols, rows;  // output columns and rows of a block
  int32_t n;           // views
  uint32_t n_blocks;   // blocks
  float lam;           // lambda_SSIM
  float inv_views;     // 1 / n
  uint64_t plane;      // floats in one partial plane (3 * all pixels)
};

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }

// the view owning block b: the last view whose first block is <= b
__device__ __forceinline__ int loss_view_of(const LossParams& P, uint32_t b) {
  int lo = 0, hi = P.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (P.v[mid].blk_off <= b) lo = mid; else hi = mid - 1;
  }
  return lo;
}

struct StripAt {
  int W, H, gx0, gy0, rows;  // image size, first output pixel, output rows
  size_t base;               // float offset of the channel plane in the packed images
};
__device__ __forceinline__ StripAt strip_at(const LossParams& P, uint32_t block) {
  const LossView& w = P.v[loss_view_of(P, block)];
  const uint32_t lb = block - w.blk_off;
  const uint32_t ch = lb / w.tiles, ti = lb % w.tiles;
  StripAt s;
  s.W = w.W;
  s.H = w.H;
  s.gx0 = (ti % w.tiles_x) * P.cols;
  s.gy0 = (ti / w.tiles_x) * P.rows;
  s.rows = min(P.rows, w.H - s.gy0);
  s.base = (size_t)w.pix_off * 3 + (size_t)ch * w.W * w.H;
  return s;
}

// 4-byte asynchronous copy global -> shared (sm_80 and later) from src + bytes;
// with size 0 (not 4) it writes zero and reads nothing, the address then only
// has to be some mapped one.
__device__ __forceinline__ void cp_async4(void* dst, const float* src, uint32_t bytes, uint32_t size) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d),
               "l"(reinterpret_cast<const char*>(src) + bytes), "r"(size)
               : "memory");
}
// element at a byte offset below 2^32 of a channel plane (a channel has fewer than 2^31 / 3 pixels)
__device__ __forceinline__ const float& at_bytes(const float* p, uint32_t bytes) {
  return *reinterpret_cast<const float*>(reinterpret_cast<const char*>(p) + bytes);
}
__device__ __forceinline__ float& at_bytes(float* p, uint32_t bytes) {
  return *reinterpret_cast<float*>(reinterpret_cast<char*>(p) + bytes);
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Shared-memory rows.  Along a row a thread sums four neighbouring columns
// (lane l: row l % 4 of the step, columns 4 (l / 4) .. + 3 of the warp's 32),
// and then takes its own column's sums of the four rows, which the warp has
// exchanged.  A quarter warp's 16-byte words (four rows by two column groups)
// must lie in eight different 16-byte slots of 128: for rows of pairs, whose
// groups are two slots apart, rows are offset by 0, 1, 4 and 5 slots; for rows
// of single values by 0, 2, 4 and 6; for rows of float4s by 0, 1, 2 and 3.
constexpr int kPairRow = 144;  // float2s from row to row of a step's pairs, before the offset
__device__ __forceinline__ int pair_row(int r) { return r * kPairRow + (r & 1) * 2 + (r >> 1) * 8; }
constexpr int kPairStep = 4 * kPairRow + 2 + 8;
constexpr int kOneRow = 168;   // floats from row to row of a step's single values
constexpr int kOneStep = 4 * kOneRow;
__device__ __forceinline__ int xpair_row(int r) { return r * 32 + (r & 1) * 2 + (r >> 1) * 8; }
constexpr int kXPair = 4 * 32 + 2 + 8;  // float2s of a warp's exchanged pairs
constexpr int kXOneRow = 40, kXOne = 4 * kXOneRow;
constexpr int kXQuadRow = 33, kXQuad = 4 * kXQuadRow;
static_assert(kLR == 4 && kPairRow >= kLW && kOneRow >= kLW, "rows of a step");

// Starts the copies of kLR input rows, from row y, of a strip with its halo
// (columns -kRad .. kLT + kRad - 1 of the strip), zero outside the image.
// copy(r, c, offset, size): row and column in the step's buffer, byte offset
// of the pixel in its channel plane, 4 (or 0, and offset 0, outside the image).
template <typename Copy>
__device__ __forceinline__ void start_rows(const StripAt& s, int y, Copy copy) {
  const int t = threadIdx.x, gx = s.gx0 - kRad + t;
  const bool ca = (unsigned)gx < (unsigned)s.W, cb = gx + kLT < s.W;
  uint32_t o = 4u * (uint32_t)(y * s.W + gx);  // wraps where it is not used
#pragma unroll
  for (int r = 0; r < kLR; ++r, o += 4u * (uint32_t)s.W) {
    const bool row = (unsigned)(y + r) < (unsigned)s.H;
    copy(r, t, row && ca ? o : 0u, row && ca ? 4u : 0u);
    if (t < 2 * kRad) copy(r, t + kLT, row && cb ? o + 4u * kLT : 0u, row && cb ? 4u : 0u);
  }
}

// The 1-D window in registers.
struct Window {
  float2 g[kRad + 1];
  __device__ __forceinline__ explicit Window(const LossParams& P) {
#pragma unroll
    for (int k = 0; k <= kRad; ++k) {
      g[k] = P.g2[k];
      asm volatile("" : "+f"(g[k].x), "+f"(g[k].y));  // held in registers: not fetched again from the parameters at each use
    }
  }
  __device__ __forceinline__ float2 tap(int k) const { return g[k <= kRad ? k : kWin - 1 - k]; }
};
// A row's sum enters the unfinished column sums; returns the finished one, of
// the row kRad above.  Each sum adds its rows from the top down.
__device__ __forceinline__ float2 enter(const Window& w, float2 (&a)[kWin - 1], float2 v) {
  const float2 out = fma2(w.tap(kWin - 1), v, a[0]);
#pragma unroll
  for (int i = 0; i < kWin - 2; ++i) a[i] = fma2(w.tap(kWin - 2 - i), v, a[i + 1]);
  a[kWin - 2] = mul2(w.tap(0), v);
  return out;
}
__device__ __forceinline__ float enter(const Window& w, float (&a)[kWin - 1], float v) {
  const float out = fmaf(w.tap(kWin - 1).x, v, a[0]);
#pragma unroll
  for (int i = 0; i < kWin - 2; ++i) a[i] = fmaf(w.tap(kWin - 2 - i).x, v, a[i + 1]);
  a[kWin - 2] = w.tap(0).x * v;
  return out;
}

__global__ void __launch_bounds__(kLT, kLossCtas)
    ssim_fwd_kernel(const __grid_constant__ LossParams P, const float* __restrict__ img,
                    const float* __restrict__ tgt, float* __restrict__ part, float2* __restrict__ bsum) {
  wait_prior_grid();
  __shared__ __align__(16) float2 sxy[2][kPairStep];          // (x, y)
  __shared__ __align__(16) float4 xq[kLT / 32][kXQuad];       // row sums of (x, y, x^2, y^2)
  __shared__ __align__(16) float xc[kLT / 32][kXOne];         // and of x y
  __shared__ float red[2][kLT / 32];
  const StripAt s = strip_at(P, blockIdx.x);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int hr = lane & 3, wc = 4 * (lane >> 2), hc = 32 * warp + wc;  // row and columns of the row sums
  const Window win(P);
  const bool own = s.gx0 + t < s.W;
  const float* xs = img + s.base;
  const float* ys = tgt + s.base;
  const size_t plane = P.plane;
  auto start = [&](int p, int y) {
    start_rows(s, y, [&](int r, int c, uint32_t o, uint32_t size) {
      cp_async4(&sxy[p][pair_row(r) + c].x, xs, o, size);
      cp_async4(&sxy[p][pair_row(r) + c].y, ys, o, size);
    });
  };
  float2 am[kWin - 1], aq[kWin - 1];  // unfinished sums of (x, y), (x^2, y^2) and x y
  float ac[kWin - 1];
#pragma unroll
  for (int i = 0; i < kWin - 1; ++i) {
    am[i] = aq[i] = make_float2(0.0f, 0.0f);
    ac[i] = 0.0f;
  }
  float ssum = 0.0f, lsum = 0.0f;
  const int n_in = s.rows + 2 * kRad;  // input rows, from gy0 - kRad
  start(0, s.gy0 - kRad);
  float* dst = part + s.base;
  const uint32_t rowb = 4u * (uint32_t)s.W;
  uint32_t o0 = 4u * (uint32_t)((s.gy0 - 2 * kRad) * s.W + s.gx0 + t);  // of the step's first output; wraps before it
  int p = 0;
  for (int b = 0; b < n_in; b += kLR, p ^= 1, o0 += kLR * rowb) {
    cp_async_wait_all();
    __syncthreads();  // the step's rows are there, and the other buffer's readers are done
    if (b + kLR < n_in) start(p ^ 1, s.gy0 - kRad + b + kLR);
    {
      float2 m[4], q[4];
      float x[4];
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        m[o] = q[o] = make_float2(0.0f, 0.0f);
        x[o] = 0.0f;
      }
      const float4* row = reinterpret_cast<const float4*>(&sxy[p][pair_row(hr) + hc]);
#pragma unroll
      for (int j = 0; j < kWin + 3; ++j) {
        const float4 w = row[j / 2];
        const float2 v = (j & 1) ? make_float2(w.z, w.w) : make_float2(w.x, w.y);
        const float2 sq = mul2(v, v);
        const float cr = v.x * v.y;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const int k = j - o;
          if (k < 0 || k >= kWin) continue;
          m[o] = fma2(win.tap(k), v, m[o]);
          q[o] = fma2(win.tap(k), sq, q[o]);
          x[o] = fmaf(win.tap(k).x, cr, x[o]);
        }
      }
      __syncwarp();  // the previous step's exchange has been read
#pragma unroll
      for (int o = 0; o < 4; ++o) xq[warp][hr * kXQuadRow + wc + o] = make_float4(m[o].x, m[o].y, q[o].x, q[o].y);
      *reinterpret_cast<float4*>(&xc[warp][hr * kXOneRow + wc]) = make_float4(x[0], x[1], x[2], x[3]);
      __syncwarp();
    }
#pragma unroll
    for (int r = 0; r < kLR; ++r) {
      if (own && b + r >= kRad && b + r < s.rows + kRad) {
        const float2 v = sxy[p][pair_row(r) + t + kRad];
        lsum += fabsf(v.x - v.y);
      }
      const float4 h = xq[warp][r * kXQuadRow + lane];
      const float2 fm = enter(win, am, make_float2(h.x, h.y)), fq = enter(win, aq, make_float2(h.z, h.w));
      const float fc = enter(win, ac, xc[warp][r * kXOneRow + lane]);
      const int out = b + r - 2 * kRad;  // output row of the strip
      if (out < 0 || out >= s.rows || !own) continue;
      const float mx = fm.x, my = fm.y, exx = fq.x, eyy = fq.y, exy = fc;
      const float A = 2.0f * mx * my + kC1;
      const float B = 2.0f * (exy - mx * my) + kC2;
      const float Cc = mx * mx + my * my + kC1;
      const float D = (exx - mx * mx) + (eyy - my * my) + kC2;
      const float icd = __fdividef(1.0f, Cc * D);
      const float S = A * B * icd;
      const float dA = B * icd, dB = A * icd, dC = -__fdividef(S, Cc), dD = -__fdividef(S, D);
      // through A (2 mu_y), B (-2 mu_y), Cc (2 mu_x) and D (-2 mu_x)
      const float s_mu = 2.0f * (my * (dA - dB) + mx * (dC - dD));
      const uint32_t o = o0 + (uint32_t)r * rowb;
      at_bytes(dst, o) = s_mu;
      at_bytes(dst + plane, o) = dD;
      at_bytes(dst + 2 * plane, o) = 2.0f * dB;
      ssum += S;
    }
  }
  // block sums (fixed shuffle tree, then the warps in order)
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    ssum += __shfl_xor_sync(0xffffffffu, ssum, d);
    lsum += __shfl_xor_sync(0xffffffffu, lsum, d);
  }
  if ((t & 31) == 0) {
    red[0][t >> 5] = ssum;
    red[1][t >> 5] = lsum;
  }
  __syncthreads();
  if (t == 0) {
    float a = 0.0f, b = 0.0f;
    for (int w = 0; w < kLT / 32; ++w) {
      a += red[0][w];
      b += red[1][w];
    }
    bsum[blockIdx.x] = make_float2(a, b);
  }
}

// The losses from the block sums, by one CTA: a warp per view in turn, its
// lanes' strided sums in a fixed shuffle tree, then the views in order
// (deterministic).  s_view: kLossMaxViews floats.
template <int NT>
__device__ __forceinline__ void loss_reduce(const LossParams& P, const float2* __restrict__ bsum,
                                            float* __restrict__ loss, float* s_view) {
  const int lane = threadIdx.x & 31;
  for (int v = threadIdx.x >> 5; v < P.n; v += NT / 32) {
    const LossView& w = P.v[v];
    const uint32_t nb = 3u * (uint32_t)w.tiles;
    float s = 0.0f, l = 0.0f;
#pragma unroll 8
    for (uint32_t i = lane; i < nb; i += 32) {
      const float2 q = bsum[w.blk_off + i];
      s += q.x;
      l += q.y;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, d);
      l += __shfl_xor_sync(0xffffffffu, l, d);
    }
    if (lane == 0) {
      const float n = 3.0f * (float)w.W * (float)w.H;
      s_view[v] = (1.0f - P.lam) * (l / n) + P.lam * (1.0f - s / n);
      loss[1 + v] = s_view[v];
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.0f;
    for (int v = 0; v < P.n; ++v) s += s_view[v];
    loss[0] = s / (float)P.n;
  }
}

// Block 0 reduces the losses; block 1 + i convolves strip i.
__global__ void __launch_bounds__(kLT, kLossCtas)
    ssim_bwd_kernel(const __grid_constant__ LossParams P, const float* __restrict__ img,
                    const float* __restrict__ tgt, const float* __restrict__ part, float* __restrict__ dL,
                    const float2* __restrict__ bsum, float* __restrict__ loss) {
  wait_prior_grid();
  __shared__ __align__(16) float2 sp[2][kPairStep];     // (S_mu, S_xx)
  __shared__ __align__(16) float sc[2][kOneStep];       // S_xy
  __shared__ __align__(16) float2 xp[kLT / 32][kXPair];  // row sums of both
  __shared__ __align__(16) float xc[kLT / 32][kXOne];
  if (blockIdx.x == 0) {
    loss_reduce<kLT>(P, bsum, loss, reinterpret_cast<float*>(sp));
    return;
  }
  const StripAt s = strip_at(P, blockIdx.x - 1);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int hr = lane & 3, wc = 4 * (lane >> 2), hc = 32 * warp + wc;
  const size_t plane = P.plane;
  const Window win(P);
  const bool own = s.gx0 + t < s.W;
  const float* ps = part + s.base;
  auto start = [&](int p, int y) {
    start_rows(s, y, [&](int r, int c, uint32_t o, uint32_t size) {
      cp_async4(&sp[p][pair_row(r) + c].x, ps, o, size);
      cp_async4(&sp[p][pair_row(r) + c].y, ps + plane, o, size);
      cp_async4(&sc[p][r * kOneRow + c], ps + 2 * plane, o, size);
    });
  };
  float2 am[kWin - 1];
  float ac[kWin - 1];
#pragma unroll
  for (int i = 0; i < kWin - 1; ++i) {
    am[i] = make_float2(0.0f, 0.0f);
    ac[i] = 0.0f;
  }
  const float n_inv = 1.0f / (3.0f * (float)s.W * (float)s.H);
  const float w1 = P.inv_views * n_inv * (1.0f - P.lam), ws = P.inv_views * n_inv * P.lam;
  const int n_in = s.rows + 2 * kRad;
  start(0, s.gy0 - kRad);
  const float* xs = img + s.base;
  const float* ys = tgt + s.base;
  float* dst = dL + s.base;
  const uint32_t rowb = 4u * (uint32_t)s.W;
  uint32_t o0 = 4u * (uint32_t)((s.gy0 - 2 * kRad) * s.W + s.gx0 + t);  // of the step's first output; wraps before it
  int p = 0;
  for (int b = 0; b < n_in; b += kLR, p ^= 1, o0 += kLR * rowb) {
    // the step's outputs' image and target values, to arrive during the sums
    float xo[kLR], yo[kLR];
#pragma unroll
    for (int r = 0; r < kLR; ++r) {
      const int out = b + r - 2 * kRad;
      const bool in = own && out >= 0 && out < s.rows;
      xo[r] = in ? at_bytes(xs, o0 + (uint32_t)r * rowb) : 0.0f;
      yo[r] = in ? at_bytes(ys, o0 + (uint32_t)r * rowb) : 0.0f;
    }
    cp_async_wait_all();
    __syncthreads();  // the step's rows are there, and the other buffer's readers are done
    if (b + kLR < n_in) start(p ^ 1, s.gy0 - kRad + b + kLR);
    {
      float2 m[4];
      float c[4];
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        m[o] = make_float2(0.0f, 0.0f);
        c[o] = 0.0f;
      }
      const float4* row = reinterpret_cast<const float4*>(&sp[p][pair_row(hr) + hc]);
      const float4* one = reinterpret_cast<const float4*>(&sc[p][hr * kOneRow + hc]);
      float4 u = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
      for (int j = 0; j < kWin + 3; ++j) {
        const float4 w = row[j / 2];
        const float2 v = (j & 1) ? make_float2(w.z, w.w) : make_float2(w.x, w.y);
        if (j % 4 == 0) u = one[j / 4];
        const float z = j % 4 == 0 ? u.x : j % 4 == 1 ? u.y : j % 4 == 2 ? u.z : u.w;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const int k = j - o;
          if (k < 0 || k >= kWin) continue;
          m[o] = fma2(win.tap(k), v, m[o]);
          c[o] = fmaf(win.tap(k).x, z, c[o]);
        }
      }
      __syncwarp();  // the previous step's exchange has been read
      float4* dst = reinterpret_cast<float4*>(&xp[warp][xpair_row(hr) + wc]);
      dst[0] = make_float4(m[0].x, m[0].y, m[1].x, m[1].y);
      dst[1] = make_float4(m[2].x, m[2].y, m[3].x, m[3].y);
      *reinterpret_cast<float4*>(&xc[warp][hr * kXOneRow + wc]) = make_float4(c[0], c[1], c[2], c[3]);
      __syncwarp();
    }
#pragma unroll
    for (int r = 0; r < kLR; ++r) {
      const float2 fm = enter(win, am, xp[warp][xpair_row(r) + lane]);
      const float fc = enter(win, ac, xc[warp][r * kXOneRow + lane]);
      const int out = b + r - 2 * kRad;
      if (out < 0 || out >= s.rows || !own) continue;
      const float x = xo[r], y = yo[r];
      const float sg = (float)(x > y) - (float)(x < y);
      // d(1 - SSIM)/dx = -dSSIM/dx
      at_bytes(dst, o0 + (uint32_t)r * rowb) = w1 * sg - ws * (fm.x + 2.0f * x * fm.y + y * fc);
    }
  }
}

// ---------------------------------------------------------------- small images
//
// A CTA per 32 x 32 tile, staged whole with its halo, both passes through
// shared memory: more arithmetic and shared-memory traffic per pixel than a
// strip, but a single step, and all tiles at once (see loss_blocks).
constexpr int kTX = 32, kTY = 32;       // output tile
constexpr int kHY = kTY + 2 * kRad;     // halo rows
constexpr int kCOff = 8;                // shared-memory column of tile column 0
constexpr int kSW = kCOff + kTX + 8;    // shared-memory row: tile columns -8 .. 39
constexpr int kTileThreads = 256;
constexpr int kTileCtas = 5;            // CTAs per SM
static_assert(kTX == kSumTile && kTY == kSumTile, "a block sum per tile");

__device__ __forceinline__ float2 tap(const LossParams& P, int k) { return P.g2[k <= kRad ? k : kWin - 1 - k]; }

// Fills the tile with its halo (rows -5 .. 36, columns -8 .. 39 of the tile)
// in shared memory, zero outside the image, with asynchronous copies: one
// warp per row, each lane two columns, every copy of the thread in flight
// before it waits.  copy(r, c, offset, in) issues the copies of one element
// (offset: of the pixel within its plane set; clamped to the tile's first
// pixel when !in).
template <typename Copy>
__device__ __forceinline__ void load_halo(const StripAt& t, Copy copy) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gxa = t.gx0 - kCOff + lane, gxb = gxa + 32;
  const bool ca = gxa >= 0 && gxa < t.W, cb = lane < kSW - 32 && gxb >= 0 && gxb < t.W;
  constexpr int kRows = (kHY + kTileThreads / 32 - 1) / (kTileThreads / 32);
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
    const int r = warp + i * (kTileThreads / 32);
    if (r < kHY) {
      const int gy = t.gy0 - kRad + r;
      const bool ry = gy >= 0 && gy < t.H;
      const size_t row = t.base + (size_t)(ry ? gy : t.gy0) * t.W;
      copy(r, lane, row + (ry && ca ? gxa : t.gx0), ry && ca);
      if (lane < kSW - 32) copy(r, lane + 32, row + (ry && cb ? gxb : t.gx0), ry && cb);
    }
  }
  cp_async_wait_all();
}

// Row pass over one halo row r: the 11-tap window sums at output columns c0
// and c0 + 1 (tile coordinates), from the 16-byte words of shared columns
// c0 + 2 .. c0 + 15 (tile columns c0 - 6 .. c0 + 7).  F receives each loaded
// column with, per output o, its tap k (or -1).
template <typename F>
__device__ __forceinline__ void row_taps(int c0, F f) {
#pragma unroll
  for (int ch = 0; ch < 7; ++ch)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int j = 2 * ch + e;  // tile column c0 - 6 + j
      const int k0 = j - 1, k1 = j - 2;
      f(c0 + 2 + 2 * ch, e, (k0 >= 0 && k0 < kWin) ? k0 : -1, (k1 >= 0 && k1 < kWin) ? k1 : -1);
    }
}

__global__ void __launch_bounds__(kTileThreads, kTileCtas)
    ssim_fwd_tile_kernel(const __grid_constant__ LossParams P, const float* __restrict__ img,
                         const float* __restrict__ tgt, float* __restrict__ part, float2* __restrict__ bsum) {
  wait_prior_grid();
  __shared__ __align__(16) float2 sxy[kHY][kSW];  // (x, y)
  __shared__ __align__(16) float2 hm[kHY][kTX];   // row sums of (x, y)
  __shared__ __align__(16) float2 hq[kHY][kTX];   // row sums of (x^2, y^2)
  __shared__ __align__(16) float hc[kHY][kTX];    // row sums of x y
  __shared__ float red[2][kTileThreads / 32];
  const StripAt t = strip_at(P, blockIdx.x);
  const int W = t.W, H = t.H;
  load_halo(t, [&](int r, int c, size_t o, bool in) {
    cp_async4(&sxy[r][c].x, img + o, 0u, in ? 4u : 0u);
    cp_async4(&sxy[r][c].y, tgt + o, 0u, in ? 4u : 0u);
  });
  __syncthreads();
  // rows: two output columns per work item, (x, y) and (x^2, y^2) in packed pairs
  for (int it = threadIdx.x; it < kHY * (kTX / 2); it += kTileThreads) {
    const int r = it / (kTX / 2), c0 = 2 * (it % (kTX / 2));
    float2 m0 = make_float2(0.0f, 0.0f), m1 = m0, q0 = m0, q1 = m0;
    float x0 = 0.0f, x1 = 0.0f;
    float4 w = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    row_taps(c0, [&](int col, int e, int k0, int k1) {
      if (e == 0) w = *reinterpret_cast<const float4*>(&sxy[r][col]);
      const float2 v = e == 0 ? make_float2(w.x, w.y) : make_float2(w.z, w.w);
      const float2 sq = mul2(v, v);
      const float cr = v.x * v.y;
      if (k0 >= 0) {
        m0 = fma2(tap(P, k0), v, m0);
        q0 = fma2(tap(P, k0), sq, q0);
        x0 = fmaf(tap(P, k0).x, cr, x0);
      }
      if (k1 >= 0) {
        m1 = fma2(tap(P, k1), v, m1);
        q1 = fma2(tap(P, k1), sq, q1);
        x1 = fmaf(tap(P, k1).x, cr, x1);
      }
    });
    *reinterpret_cast<float4*>(&hm[r][c0]) = make_float4(m0.x, m0.y, m1.x, m1.y);
    *reinterpret_cast<float4*>(&hq[r][c0]) = make_float4(q0.x, q0.y, q1.x, q1.y);
    *reinterpret_cast<float2*>(&hc[r][c0]) = make_float2(x0, x1);
  }
  __syncthreads();
  // columns: four output rows per thread
  const int c = threadIdx.x % kTX, r0 = 4 * (threadIdx.x / kTX);
  float2 am[4], aq[4];
  float ac[4];
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    am[o] = aq[o] = make_float2(0.0f, 0.0f);
    ac[o] = 0.0f;
  }
#pragma unroll
  for (int j = 0; j < kWin + 3; ++j) {
    const float2 m = hm[r0 + j][c], q = hq[r0 + j][c];
    const float x = hc[r0 + j][c];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const int k = j - o;
      if (k < 0 || k >= kWin) continue;
      am[o] = fma2(tap(P, k), m, am[o]);
      aq[o] = fma2(tap(P, k), q, aq[o]);
      ac[o] = fmaf(tap(P, k).x, x, ac[o]);
    }
  }
  float ssum = 0.0f, lsum = 0.0f;
  const size_t plane = P.plane;
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    const int r = r0 + o;
    const int gx = t.gx0 + c, gy = t.gy0 + r;
    if (gx >= W || gy >= H) continue;
    const float mx = am[o].x, my = am[o].y, exx = aq[o].x, eyy = aq[o].y, exy = ac[o];
    const float A = 2.0f * mx * my + kC1;
    const float B = 2.0f * (exy - mx * my) + kC2;
    const float Cc = mx * mx + my * my + kC1;
    const float D = (exx - mx * mx) + (eyy - my * my) + kC2;
    const float icd = __fdividef(1.0f, Cc * D);
    const float S = A * B * icd;
    const float dA = B * icd, dB = A * icd, dC = -__fdividef(S, Cc), dD = -__fdividef(S, D);
    // through A (2 mu_y), B (-2 mu_y), Cc (2 mu_x) and D (-2 mu_x)
    const float s_mu = 2.0f * (my * (dA - dB) + mx * (dC - dD));
    const size_t idx = t.base + (size_t)gy * W + gx;
    part[idx] = s_mu;
    part[plane + idx] = dD;
    part[2 * plane + idx] = 2.0f * dB;
    ssum += S;
    const float2 xy = sxy[r + kRad][c + kCOff];
    lsum += fabsf(xy.x - xy.y);
  }
  // block sums (fixed shuffle tree, then the warps in order)
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    ssum += __shfl_xor_sync(0xffffffffu, ssum, d);
    lsum += __shfl_xor_sync(0xffffffffu, lsum, d);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = ssum;
    red[1][threadIdx.x >> 5] = lsum;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float a = 0.0f, b = 0.0f;
    for (int w = 0; w < kTileThreads / 32; ++w) {
      a += red[0][w];
      b += red[1][w];
    }
    bsum[blockIdx.x] = make_float2(a, b);
  }
}

__global__ void __launch_bounds__(kTileThreads, kTileCtas)
    ssim_bwd_tile_kernel(const __grid_constant__ LossParams P, const float* __restrict__ img,
                         const float* __restrict__ tgt, const float* __restrict__ part, float* __restrict__ dL,
                         const float2* __restrict__ bsum, float* __restrict__ loss) {
  wait_prior_grid();
  __shared__ __align__(16) float2 sp[kHY][kSW];  // (S_mu, S_xx)
  __shared__ __align__(16) float sc[kHY][kSW];   // S_xy
  __shared__ __align__(16) float2 hp[kHY][kTX];
  __shared__ __align__(16) float hs[kHY][kTX];
  if (blockIdx.x == 0) {
    loss_reduce<kTileThreads>(P, bsum, loss, reinterpret_cast<float*>(sp));
    return;
  }
  const StripAt t = strip_at(P, blockIdx.x - 1);
  const int W = t.W, H = t.H;
  const size_t plane = P.plane;
  // this thread's four outputs (column c, rows r0 .. r0 + 3): their image and
  // target values are loaded first, to arrive during the passes
  const int c = threadIdx.x % kTX, r0 = 4 * (threadIdx.x / kTX);
  float xo[4], yo[4];
  size_t io[4];
  bool ok[4];
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    const int gx = t.gx0 + c, gy = t.gy0 + r0 + o;
    ok[o] = gx < W && gy < t.H;
    io[o] = t.base + (size_t)(ok[o] ? gy : 0) * W + (ok[o] ? gx : 0);
    xo[o] = ok[o] ? img[io[o]] : 0.0f;
    yo[o] = ok[o] ? tgt[io[o]] : 0.0f;
  }
  load_halo(t, [&](int r, int cc, size_t o, bool in) {
    cp_async4(&sp[r][cc].x, part + o, 0u, in ? 4u : 0u);
    cp_async4(&sp[r][cc].y, part + plane + o, 0u, in ? 4u : 0u);
    cp_async4(&sc[r][cc], part + 2 * plane + o, 0u, in ? 4u : 0u);
  });
  __syncthreads();
  for (int it = threadIdx.x; it < kHY * (kTX / 2); it += kTileThreads) {
    const int r = it / (kTX / 2), c0 = 2 * (it % (kTX / 2));
    float2 a0 = make_float2(0.0f, 0.0f), a1 = a0;
    float b0 = 0.0f, b1 = 0.0f;
    float4 w = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float2 z = make_float2(0.0f, 0.0f);
    row_taps(c0, [&](int col, int e, int k0, int k1) {
      if (e == 0) {
        w = *reinterpret_cast<const float4*>(&sp[r][col]);
        z = *reinterpret_cast<const float2*>(&sc[r][col]);
      }
      const float2 v = e == 0 ? make_float2(w.x, w.y) : make_float2(w.z, w.w);
      const float u = e == 0 ? z.x : z.y;
      if (k0 >= 0) {
        a0 = fma2(tap(P, k0), v, a0);
        b0 = fmaf(tap(P, k0).x, u, b0);
      }
      if (k1 >= 0) {
        a1 = fma2(tap(P, k1), v, a1);
        b1 = fmaf(tap(P, k1).x, u, b1);
      }
    });
    *reinterpret_cast<float4*>(&hp[r][c0]) = make_float4(a0.x, a0.y, a1.x, a1.y);
    *reinterpret_cast<float2*>(&hs[r][c0]) = make_float2(b0, b1);
  }
  __syncthreads();
  float2 am[4];
  float ab[4];
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    am[o] = make_float2(0.0f, 0.0f);
    ab[o] = 0.0f;
  }
#pragma unroll
  for (int j = 0; j < kWin + 3; ++j) {
    const float2 m = hp[r0 + j][c];
    const float u = hs[r0 + j][c];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const int k = j - o;
      if (k < 0 || k >= kWin) continue;
      am[o] = fma2(tap(P, k), m, am[o]);
      ab[o] = fmaf(tap(P, k).x, u, ab[o]);
    }
  }
  const float n_inv = 1.0f / (3.0f * (float)W * (float)H);
  const float w1 = P.inv_views * n_inv * (1.0f - P.lam), ws = P.inv_views * n_inv * P.lam;
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    if (!ok[o]) continue;
    const float x = xo[o], y = yo[o];
    const float sg = (float)(x > y) - (float)(x < y);
    // d(1 - SSIM)/dx = -dSSIM/dx
    dL[io[o]] = w1 * sg - ws * (am[o].x + 2.0f * x * am[o].y + y * ab[o]);
  }
}

// ---------------------------------------------------------------------------
// Adam
// ---------------------------------------------------------------------------

constexpr int kAdamMaxPlanes = 64;
struct AdamParams {
  float lr[kAdamMaxPlanes];
  float l1[kAdamMaxPlanes];
  int32_t act[kAdamMaxPlanes];
  int32_t noise_row[kAdamMaxPlanes];
  int64_t P;
  int32_t K;
  float b1, b2, eps, bc1, bc2, leps;  // bc = 1 / (1 - beta^t)
};

__device__ __forceinline__ float activate(float r, int act) {
  if (act == UBS_ACT_SIGMOID) return 1.0f / (1.0f + expf(-r));
  if (act == UBS_ACT_EXP) return expf(r);
  return r;
}

__device__ __forceinline__ void adam_one(const AdamParams& A, int k, float& r, float& a, float g, float& m,
                                         float& v, float noise) {
  const int act = A.act[k];
  const float a0 = activate(r, act);
  g += A.l1[k] * ((float)(a0 > 0.0f) - (float)(a0 < 0.0f));
  if (act == UBS_ACT_SIGMOID) g *= a0 * (1.0f - a0);
  else if (act == UBS_ACT_EXP) g *= a0;
  m = fmaf(A.b1, m, (1.0f - A.b1) * g);
  v = fmaf(A.b2, v, (1.0f - A.b2) * g * g);
  r -= A.lr[k] * (m * A.bc1) / (sqrtf(v * A.bc2) + A.eps);
  r = fmaf(A.leps, noise, r);
  a = activate(r, act);
}

// The plane of element e < K P: an estimate in float, at most one off (e / P
// is below 64), corrected; a 64-bit division costs more than the update.
__device__ __forceinline__ int plane_of(int64_t e, int64_t P, float inv_p) {
  int k = (int)((float)e * inv_p);
  if (e < (int64_t)k * P) --k;
  if (e >= (int64_t)(k + 1) * P) ++k;
  return k;
}

// The K P elements as one array, four to a thread: with every array on a
// 16-byte boundary as 16-byte words whatever P is.  Where P is a multiple of
// four and the noise lies on such a boundary too (kAdamPlaneWords), a word is
// of one plane and the noise is read by words.  Else (kAdamWords) a word can
// straddle two planes, so each element takes its own plane's constants, and
// the noise, whose rows start anywhere against the words, is read by elements.
// Bound by HBM: 500,003 x 35 parameters 104 us by single elements (5.5 TB/s),
// 88 us (6.4 TB/s) by words; 500,000 x 35 with noise 92.7 us by words, 91.1 by
// words within planes, x 20 57.5 and 55.7.
enum AdamForm { kAdamElements, kAdamWords, kAdamPlaneWords };
template <AdamForm FORM>
__global__ void __launch_bounds__(256)
    adam_kernel(const __grid_constant__ AdamParams A, float* __restrict__ raw, float* __restrict__ act,
                const float* __restrict__ grad, float* __restrict__ m, float* __restrict__ v,
                const float* __restrict__ noise) {
  wait_prior_grid();
  const int64_t n = (int64_t)A.K * A.P;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const float inv_p = 1.0f / (float)A.P;
  auto noise_at = [&](int k, int64_t e) {
    const int row = A.noise_row[k];
    return row >= 0 ? noise[(int64_t)row * A.P + (e - (int64_t)k * A.P)] : 0.0f;
  };
  auto one = [&](int64_t e) {
    const int k = plane_of(e, A.P, inv_p);
    const float z = noise_at(k, e);
    float r = raw[e], mm = m[e], vv = v[e], a;
    adam_one(A, k, r, a, grad[e], mm, vv, z);
    raw[e] = r;
    act[e] = a;
    m[e] = mm;
    v[e] = vv;
  };
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if constexpr (FORM != kAdamElements) {
    for (int64_t q = t0; q < n / 4; q += stride) {
      const int64_t e = 4 * q;
      float4 r = reinterpret_cast<float4*>(raw)[q];
      const float4 g = reinterpret_cast<const float4*>(grad)[q];
      float4 mm = reinterpret_cast<float4*>(m)[q];
      float4 vv = reinterpret_cast<float4*>(v)[q];
      float4 a;
      const int k = plane_of(e, A.P, inv_p);
      if constexpr (FORM == kAdamPlaneWords) {
        const int row = A.noise_row[k];
        float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (row >= 0) z = reinterpret_cast<const float4*>(noise + (int64_t)row * A.P)[(e - (int64_t)k * A.P) / 4];
        adam_one(A, k, r.x, a.x, g.x, mm.x, vv.x, z.x);
        adam_one(A, k, r.y, a.y, g.y, mm.y, vv.y, z.y);
        adam_one(A, k, r.z, a.z, g.z, mm.z, vv.z, z.z);
        adam_one(A, k, r.w, a.w, g.w, mm.w, vv.w, z.w);
      } else {
        const int64_t left = (int64_t)(k + 1) * A.P - e;  // elements of the word in plane k, if below 4
        // (planes of fewer than three elements: the last one's may lie two on)
        auto plane = [&](int i) { return left > i ? k : plane_of(e + i, A.P, inv_p); };
        const int k1 = plane(1), k2 = plane(2), k3 = plane(3);
        adam_one(A, k, r.x, a.x, g.x, mm.x, vv.x, noise_at(k, e));
        adam_one(A, k1, r.y, a.y, g.y, mm.y, vv.y, noise_at(k1, e + 1));
        adam_one(A, k2, r.z, a.z, g.z, mm.z, vv.z, noise_at(k2, e + 2));
        adam_one(A, k3, r.w, a.w, g.w, mm.w, vv.w, noise_at(k3, e + 3));
      }
      reinterpret_cast<float4*>(raw)[q] = r;
      reinterpret_cast<float4*>(act)[q] = a;
      reinterpret_cast<float4*>(m)[q] = mm;
      reinterpret_cast<float4*>(v)[q] = vv;
    }
    if (t0 < n % 4) one(n - n % 4 + t0);
  } else {
    for (int64_t e = t0; e < n; e += stride) one(e);
  }
}

// Whether the images go by tiles: where they are few (fewer than 2.5 waves of
// tile CTAs), as a strip's many steps are then a latency that nothing hides, or
// narrow, as a strip's unused columns cost more than its saved arithmetic
// gains.  Both kernels by tiles / strips, us: one 256 x 192 image 11 / 24, 400
// x 301 17 / 26, 800 x 600 36 / 38; two of them (2850 tiles) 58 / 58, three 87
// / 77; 640 x 360 two (1440) 36 / 38, three (2160) 48 / 46, eight 118 / 89; 256
// of 64 x 64 (strips of twice the tiles' pixels) 67 / 103, sixteen of 130 x
// 1000 (1.56 times) 151 / 181, eight of 260 x 1000 (1.30) 138 / 140, eight of
// 400 x 301 (1.16) 64 / 67, one of 1352 x 1014 83 / 73.  Images of a few rows,
// most of a tile's empty, go by strips of as few steps: 4000 x 5 15 / 13.
bool use_tiles(uint64_t tiles, uint64_t strip_px, uint64_t tile_px, int sms) {
  if (4 * strip_px < tile_px) return false;
  return 2 * tiles < 5ull * kTileCtas * sms || 4 * strip_px > 5 * tile_px;
}

int sm_count() {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// Sizes and, with P, the blocks of the two kernels on a device of `sms` SMs.
bool loss_blocks(int32_t n, const int32_t* w, const int32_t* h, int sms, LossParams* P, size_t* ws) {
  if (n < 1 || n > kLossMaxViews || !w || !h) return false;
  uint64_t pix = 0, sums = 0, strip_px = 0, tile_px = 0;
  for (int i = 0; i < n; ++i) {
    if (w[i] < 1 || h[i] < 1 || w[i] > 65535 || h[i] > 65535) return false;
    pix += (uint64_t)w[i] * h[i];
    sums += 3ull * ((w[i] + kSumTile - 1) / kSumTile) * ((h[i] + kSumTile - 1) / kSumTile);
    strip_px += 3ull * ((w[i] + kLT - 1) / kLT) * kLT * h[i];
    tile_px += 3ull * ((w[i] + kTX - 1) / kTX) * kTX * ((h[i] + kTY - 1) / kTY) * kTY;
    if (pix > 0x7fffffffull / 3 || sums > 0x7fffffffull) return false;
  }
  *ws = align256(3 * 3 * pix * sizeof(float)) + align256(sums * sizeof(float2));
  if (!P) return true;
  if (use_tiles(sums, strip_px, tile_px, sms)) {
    P->cols = kTX;
    P->rows = kTY;
  } else {
    // The strips' height: a multiple of the step, between kMinRows (each strip
    // also walks 2 kRad halo rows: 16 and 24 rows took 150 and 148 us for a
    // training step at 800 x 600, 32 took 147) and kMaxRows, and in between the
    // least for which all CTAs, the backward's reducing one too, are resident
    // at once (1920 x 1080 with five strips too many 112 us, so 97); as
    // kMinRows >= kSumTile there is a block sum for each
    static_assert(kMinRows >= kSumTile && kMinRows % kLR == 0 && kLT >= kSumTile, "a block sum per strip");
    uint64_t rows = kMinRows;
    auto blocks = [&](uint64_t r) {
      uint64_t k = 1;
      for (int i = 0; i < n; ++i) k += 3ull * ((w[i] + kLT - 1) / kLT) * ((h[i] + r - 1) / r);
      return k;
    };
    while (rows < kMaxRows && blocks(rows) > (uint64_t)sms * kLossCtas) rows += kLR;
    P->cols = kLT;
    P->rows = (int32_t)rows;
  }
  uint64_t blk = 0, at = 0;
  for (int i = 0; i < n; ++i) {
    LossView& v = P->v[i];
    v.W = w[i];
    v.H = h[i];
    v.tiles_x = (w[i] + P->cols - 1) / P->cols;
    v.tiles = v.tiles_x * ((h[i] + P->rows - 1) / P->rows);
    v.pix_off = (uint32_t)at;
    v.blk_off = (uint32_t)blk;
    at += (uint64_t)w[i] * h[i];
    blk += 3ull * v.tiles;
  }
  P->n_blocks = (uint32_t)blk;
  P->n = n;
  P->plane = 3 * pix;
  return true;
}

}  // namespace
}  // namespace ubs

using namespace ubs;

extern "C" size_t ubs_loss_workspace_size(int32_t n_views, const int32_t* widths, const int32_t* heights) {
  size_t ws = 0;
  return loss_blocks(n_views, widths, heights, 0, nullptr, &ws) ? ws : 0;
}

extern "C" ubs_status ubs_image_loss(int32_t n_views, const int32_t* widths, const int32_t* heights,
                                     const float* image, const float* target, float lambda_ssim, float* dL_dimage,
                                     float* loss, void* workspace, size_t workspace_bytes, cudaStream_t stream) {
  ubs::TraceRange trace_("ubs_image_loss");
  size_t need = 0;
  if (!loss_blocks(n_views, widths, heights, 0, nullptr, &need)) return UBS_ERR_INVALID_ARG;
  if (!image || !target || !dL_dimage || !loss || !workspace) return UBS_ERR_INVALID_ARG;
  if (!(lambda_ssim >= 0.0f && lambda_ssim <= 1.0f)) return UBS_ERR_INVALID_ARG;
  if (((uintptr_t)workspace & 255u) != 0) return UBS_ERR_ALIGNMENT;
  if (((uintptr_t)image | (uintptr_t)target | (uintptr_t)dL_dimage | (uintptr_t)loss) & 3u) return UBS_ERR_ALIGNMENT;
  if (workspace_bytes < need) return UBS_ERR_WORKSPACE;
  LossParams p;
  memset(&p, 0, sizeof(p));
  loss_blocks(n_views, widths, heights, sm_count(), &p, &need);
  // the 1-D window: exp(-(i - 5)^2 / (2 * 1.5^2)), normalised to sum 1
  double g[kWin], s = 0.0;
  for (int i = 0; i < kWin; ++i) {
    g[i] = exp(-(double)((i - kRad) * (i - kRad)) / (2.0 * 1.5 * 1.5));
    s += g[i];
  }
  for (int i = 0; i <= kRad; ++i) p.g2[i] = make_float2((float)(g[i] / s), (float)(g[i] / s));
  p.lam = lambda_ssim;
  p.inv_views = 1.0f / (float)n_views;
  char* ws = (char*)workspace;
  float* part = (float*)ws;
  float2* bsum = (float2*)(ws + align256(3 * p.plane * sizeof(float)));
  const bool tiles = p.cols == kTX;
  const dim3 block(tiles ? kTileThreads : kLT);
  cudaError_t e = launch_dependent(tiles ? ssim_fwd_tile_kernel : ssim_fwd_kernel, dim3(p.n_blocks), block, 0, stream,
                                   p, image, target, part, bsum);
  if (e == cudaSuccess)
    e = launch_dependent(tiles ? ssim_bwd_tile_kernel : ssim_bwd_kernel, dim3(p.n_blocks + 1), block, 0, stream, p,
                         image, target, (const float*)part, dL_dimage, (const float2*)bsum, loss);
  return e == cudaSuccess ? UBS_OK : UBS_ERR_CUDA;
}

extern "C" ubs_status ubs_adam_step(int32_t K, int64_t P, const ubs_adam_plane* planes, const ubs_adam_config* cfg,
                                    float* raw, float* act_out, const float* grad, float* m, float* v,
                                    const float* noise, cudaStream_t stream) {
  ubs::TraceRange trace_("ubs_adam_step");
  if (K < 1 || K > kAdamMaxPlanes || P < 0 || !planes || !cfg) return UBS_ERR_INVALID_ARG;
  if (P == 0) return UBS_OK;
  if (!raw || !act_out || !grad || !m || !v || raw == act_out) return UBS_ERR_INVALID_ARG;
  if (cfg->step < 1 || !(cfg->beta1 >= 0.0f && cfg->beta1 < 1.0f) || !(cfg->beta2 >= 0.0f && cfg->beta2 < 1.0f) ||
      !(cfg->eps >= 0.0f))
    return UBS_ERR_INVALID_ARG;
  AdamParams A;
  memset(&A, 0, sizeof(A));
  bool any_noise = false;
  for (int k = 0; k < K; ++k) {
    const ubs_adam_plane& q = planes[k];
    if (q.activation < UBS_ACT_IDENTITY || q.activation > UBS_ACT_EXP || !(q.lr >= 0.0f)) return UBS_ERR_INVALID_ARG;
    A.lr[k] = q.lr;
    A.l1[k] = q.l1_weight;
    A.act[k] = q.activation;
    A.noise_row[k] = q.noise_row < 0 ? -1 : q.noise_row;
    any_noise = any_noise || q.noise_row >= 0;
  }
  if (any_noise && !noise) return UBS_ERR_INVALID_ARG;
  const uintptr_t all = (uintptr_t)raw | (uintptr_t)act_out | (uintptr_t)grad | (uintptr_t)m | (uintptr_t)v |
                        (uintptr_t)(noise ? noise : raw);
  if (all & 3u) return UBS_ERR_ALIGNMENT;
  A.P = P;
  A.K = K;
  A.b1 = cfg->beta1;
  A.b2 = cfg->beta2;
  A.eps = cfg->eps;
  A.bc1 = (float)(1.0 / (1.0 - pow((double)cfg->beta1, (double)cfg->step)));
  A.bc2 = (float)(1.0 / (1.0 - pow((double)cfg->beta2, (double)cfg->step)));
  A.leps = cfg->lambda_eps;
  // the words' arrays; of the noise only the words within planes ask it
  const bool vec = (((uintptr_t)raw | (uintptr_t)act_out | (uintptr_t)grad | (uintptr_t)m | (uintptr_t)v) & 15u) == 0;
  const AdamForm form = !vec ? kAdamElements : P % 4 == 0 && ((uintptr_t)noise & 15u) == 0 ? kAdamPlaneWords : kAdamWords;
  const int64_t units = vec ? (int64_t)K * P / 4 + 1 : (int64_t)K * P;
  const int sms = sm_count();
  const int64_t want = (units + 255) / 256;
  const unsigned grid = (unsigned)(want < (int64_t)sms * 8 ? want : (int64_t)sms * 8);
  const auto kernel = form == kAdamElements ? adam_kernel<kAdamElements>
                      : form == kAdamWords  ? adam_kernel<kAdamWords>
                                            : adam_kernel<kAdamPlaneWords>;
  const cudaError_t e = launch_dependent(kernel, dim3(grid), dim3(256), 0, stream, A, raw, act_out, grad, m, v, noise);
  return e == cudaSuccess ? UBS_OK : UBS_ERR_CUDA;
}
