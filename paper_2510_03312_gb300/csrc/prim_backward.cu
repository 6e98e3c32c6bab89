// prim_backward.cu -- G2: chain the per-record screen gradients back to the
// primitive parameters (math in prim_backward.cuh).
//
// One thread per primitive (scenes with one view: every primitive for N = 3,
// the drawn ones of its CTA's range for N > 3; with several: the list of
// primitives some view sees, built by preprocess); it
// rebuilds the view-independent quantities once, walks its visible views
// accumulating in registers, and writes every parameter gradient once: no
// atomics and a deterministic sum over views.
#include "kernels.cuh"
#include "prim_backward.cuh"

namespace ubs {

namespace {

template <int C>
__device__ __forceinline__ void load_prim_b(const SceneDev& sc, int64_t p, PrimIn<C>& in) {
  const int64_t P = sc.P;
  for (int i = 0; i < 3; ++i) in.mx[i] = __ldg(sc.mean_x + i * P + p);
  const int nr = sc.rot_mode == 0 ? 4 : 3;
  for (int i = 0; i < 4; ++i) in.rot[i] = i < nr ? __ldg(sc.rot + i * P + p) : 0.0f;
  for (int i = 0; i < 3; ++i) in.s[i] = __ldg(sc.scale_x + i * P + p);
  for (int i = 0; i < 1 + C; ++i) in.b[i] = __ldg(sc.b + i * P + p);
  in.o = __ldg(sc.opacity + p);
  if constexpr (C > 0) {
    for (int i = 0; i < C; ++i) in.mq[i] = __ldg(sc.mean_q + i * P + p);
    for (int i = 0; i < 3 * C; ++i) in.lqx[i] = __ldg(sc.L_qx + i * P + p);
    for (int i = 0; i < C * (C + 1) / 2; ++i) in.lq[i] = __ldg(sc.L_q + i * P + p);
  }
}

// Scenes of N = 3 with one view: a thread per primitive; most are drawn, and an
// undrawn one costs little.  Held to 72 registers (7 CTAs per SM): bound by
// memory latency, it gains more from occupancy than it loses to a few spills to
// L1 (63.5 us unbounded, 53.7 at 6 CTAs, 51.9 at 7 on the 1M-primitive view; 8
// gained nothing more).
__global__ void __launch_bounds__(128, 7) prim_backward_kernel(SceneDev sc, SceneGradDev gr, int view,
                                                               const ViewDev* __restrict__ views, CfgDev cfg,
                                                               const uint32_t* __restrict__ tiles,
                                                               const float4* __restrict__ g2d) {
  wait_prior_grid();
  __shared__ ViewDev s_view;
  if (threadIdx.x == 0) s_view = views[view];
  __syncthreads();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= sc.P) return;
  PrimIn<0> in;
  load_prim_b<0>(sc, p, in);
  PrimVI<0> vi;
  prim_stage<0>(in, sc.rot_mode, vi);
  PrimAcc<0> acc;
  acc_zero<0>(acc);
  const uint32_t r = s_view.rec_off + (uint32_t)p;
  if (tiles[r] != 0) {
    const float4 a = g2d[3 * (size_t)r], b = g2d[3 * (size_t)r + 1], c = g2d[3 * (size_t)r + 2];
    const float g[10] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y};
    prim_backward_view<0>(in, vi, s_view, cfg, g, acc);
  }
  PrimGrad<0> out;
  prim_backward_final<0>(in, vi, sc.rot_mode, acc, out);
  const int64_t P = sc.P;
  // written, or added to the caller's running sum (UBS_FLAG_ACCUMULATE_GRADS)
  const bool add = (cfg.flags & 4) != 0;
  auto put = [&](float* dst, float v) { *dst = add ? *dst + v : v; };
  for (int i = 0; i < 3; ++i) put(gr.mean_x + i * P + p, out.mx[i]);
  const int nr = sc.rot_mode == 0 ? 4 : 3;
  for (int i = 0; i < nr; ++i) put(gr.rot + i * P + p, out.rot[i]);
  for (int i = 0; i < 3; ++i) put(gr.scale_x + i * P + p, out.s[i]);
  put(gr.b + p, out.b[0]);
  put(gr.opacity + p, out.o);
  for (int i = 0; i < 3; ++i) put(gr.rgb + i * P + p, out.rgb[i]);
}

// Scenes with query dimensions and one view: one CTA per `prims` consecutive
// primitives.  It lists those the view draws (their visibility bits) in shared
// memory and gives each thread listed ones, whose parameters lie close
// together; then it writes zero gradients for the others (unless
// accumulating).  The query culls most records (7% drawn), on which a thread
// per primitive spent its loads and arithmetic all the same (200K N=6
// primitives: 40 us; 17 us so).  Scenes with several views draw most primitives
// in some view: there the list of the whole scene (prim_backward_listed_kernel)
// balances better (16 views of 500K N=6 primitives: 11 + 98 us, this form 144).
// How many are drawn is not known at the launch.  Where few are, a CTA's time
// is one round's latency and long ranges win; where nearly all are, a long
// range takes several rounds, and a grid that ends in a nearly empty wave waits
// for all of them.  So the range is the longest (128, 256, 384 or 512) whose
// rounds, with every primitive drawn, number at most 5/4 of the fewest that any
// length gives.  Whole step of one 640x360 view by ranges of 128 / 256 / 512,
// us (a thread per primitive before): N=7 30K primitives, 1% drawn 48 / 48 / 48
// (56), 86% drawn 107 / 113 / 124 (116); 60K 57 / 52 / 53 (65) and 176 / 176 /
// 187 (185); 160K 75 / 67 / 65 (97) and 343 / 349 / 366 (343); 300K 106 / 93 /
// 81 (142) and 416 / 413 / 414 (423); N=6 60K, 6% drawn 56 / 56 / 56 (69), 92%
// drawn 181 / 185 / 198 (193); 200K 91 / 87 / 83 (120) and 304 / 310 / 308
// (329).
constexpr int kPbThreads = 128;
constexpr int kPbPrims = 512, kPbWords = kPbPrims / 32;
inline int pb_prims(int N, int64_t P) {
  const int64_t slots = 152 * (N == 7 ? 2 : 4);  // 205 registers a thread, 128
  auto rounds = [&](int64_t r) { return r * (((P + r * kPbThreads - 1) / (r * kPbThreads) + slots - 1) / slots); };
  int64_t least = rounds(1);
  int r = kPbPrims / kPbThreads;
  for (int i = 2; i <= r; ++i) least = rounds(i) < least ? rounds(i) : least;
  while (r > 1 && 4 * rounds(r) > 5 * least) --r;
  return r * kPbThreads;
}
template <int C>
__global__ void __launch_bounds__(kPbThreads, C == 3 ? 4 : 1) prim_backward_drawn_kernel(
    SceneDev sc, SceneGradDev gr, ViewList vl, const ViewDev* __restrict__ views, CfgDev cfg,
    const uint32_t* __restrict__ vis_mask, const float4* __restrict__ g2d, int prims) {
  wait_prior_grid();
  __shared__ ViewDev s_view;
  __shared__ uint32_t s_any[kPbWords], s_first[kPbWords + 1];
  __shared__ uint16_t s_list[kPbPrims];
  const int64_t P = sc.P, p0 = (int64_t)blockIdx.x * prims;
  const uint32_t w0 = (uint32_t)(p0 >> 5), n_words = (uint32_t)min((int64_t)(prims / 32), (P + 31) / 32 - (int64_t)w0);
  const ViewDev& vd = views[vl.idx[0]];
  if (threadIdx.x < kPbWords) s_any[threadIdx.x] = threadIdx.x < n_words ? vis_mask[vd.mask_off + w0 + threadIdx.x] : 0u;
  if (threadIdx.x == 0) s_view = vd;
  __syncthreads();
  if (threadIdx.x < 32) {  // the first list position of each word
    const uint32_t n = threadIdx.x < kPbWords ? __popc(s_any[threadIdx.x]) : 0u;
    uint32_t x = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
      if ((int)threadIdx.x >= d) x += y;
    }
    if (threadIdx.x < kPbWords) s_first[threadIdx.x] = x - n;
    if (threadIdx.x == kPbWords - 1) s_first[kPbWords] = x;
  }
  __syncthreads();
  const bool add = (cfg.flags & 4) != 0;  // add to the caller's running sum (UBS_FLAG_ACCUMULATE_GRADS)
  const int nr = sc.rot_mode == 0 ? 4 : 3;
  for (int i = threadIdx.x; i < prims; i += kPbThreads) {
    const uint32_t any = s_any[i >> 5], bit = 1u << (i & 31);
    if (any & bit) s_list[s_first[i >> 5] + __popc(any & (bit - 1u))] = (uint16_t)i;
  }
  __syncthreads();
  const uint32_t n_items = s_first[kPbWords];
  auto put = [&](float* dst, float v) { *dst = add ? *dst + v : v; };
  for (uint32_t i = threadIdx.x; i < n_items; i += kPbThreads) {
    const uint32_t l = s_list[i];
    const int64_t p = p0 + l;
    PrimIn<C> in;
    load_prim_b<C>(sc, p, in);
    PrimVI<C> vi;
    prim_stage<C>(in, sc.rot_mode, vi);
    PrimAcc<C> acc;
    acc_zero<C>(acc);
    const uint32_t r = s_view.rec_off + (uint32_t)p;
    const float4 a = g2d[3 * (size_t)r], b = g2d[3 * (size_t)r + 1], c = g2d[3 * (size_t)r + 2];
    const float g[10] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y};
    prim_backward_view<C>(in, vi, s_view, cfg, g, acc);
    PrimGrad<C> out;
    prim_backward_final<C>(in, vi, sc.rot_mode, acc, out);
    for (int j = 0; j < 3; ++j) put(gr.mean_x + j * P + p, out.mx[j]);
    for (int j = 0; j < nr; ++j) put(gr.rot + j * P + p, out.rot[j]);
    for (int j = 0; j < 3; ++j) put(gr.scale_x + j * P + p, out.s[j]);
    for (int j = 0; j < 1 + C; ++j) put(gr.b + j * P + p, out.b[j]);
    put(gr.opacity + p, out.o);
    for (int j = 0; j < 3; ++j) put(gr.rgb + j * P + p, out.rgb[j]);
    if constexpr (C > 0) {
      for (int j = 0; j < C; ++j) put(gr.mean_q + j * P + p, out.mq[j]);
      for (int j = 0; j < 3 * C; ++j) put(gr.L_qx + j * P + p, out.lqx[j]);
      for (int j = 0; j < C * (C + 1) / 2; ++j) put(gr.L_q + j * P + p, out.lq[j]);
    }
  }
  if (add) return;
#pragma unroll 1
  for (int i = threadIdx.x; i < prims; i += kPbThreads) {
    const int64_t p = p0 + i;
    if (p >= P || ((s_any[i >> 5] >> (i & 31)) & 1u)) continue;
    for (int j = 0; j < 3; ++j) gr.mean_x[j * P + p] = 0.0f;
    for (int j = 0; j < nr; ++j) gr.rot[j * P + p] = 0.0f;
    for (int j = 0; j < 3; ++j) gr.scale_x[j * P + p] = 0.0f;
    for (int j = 0; j < 1 + C; ++j) gr.b[j * P + p] = 0.0f;
    gr.opacity[p] = 0.0f;
    for (int j = 0; j < 3; ++j) gr.rgb[j * P + p] = 0.0f;
    if constexpr (C > 0) {
      for (int j = 0; j < C; ++j) gr.mean_q[j * P + p] = 0.0f;
      for (int j = 0; j < 3 * C; ++j) gr.L_qx[j * P + p] = 0.0f;
      for (int j = 0; j < C * (C + 1) / 2; ++j) gr.L_q[j * P + p] = 0.0f;
    }
  }
}

// Zeroes one scene's gradient planes (the primitives that no view sees keep
// these zeros; the others are overwritten by prim_backward_listed_kernel).
__global__ void __launch_bounds__(256) zero_scene_grads_kernel(SceneGradDev gr, int64_t P, int C, int nr) {
  wait_prior_grid();
  const int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (p >= P) return;
  for (int i = 0; i < 3; ++i) gr.mean_x[i * P + p] = 0.0f;
  for (int i = 0; i < nr; ++i) gr.rot[i * P + p] = 0.0f;
  for (int i = 0; i < 3; ++i) gr.scale_x[i * P + p] = 0.0f;
  for (int i = 0; i < 1 + C; ++i) gr.b[i * P + p] = 0.0f;
  gr.opacity[p] = 0.0f;
  for (int i = 0; i < 3; ++i) gr.rgb[i * P + p] = 0.0f;
  for (int i = 0; i < C; ++i) gr.mean_q[i * P + p] = 0.0f;
  for (int i = 0; i < 3 * C; ++i) gr.L_qx[i * P + p] = 0.0f;
  for (int i = 0; i < C * (C + 1) / 2; ++i) gr.L_q[i * P + p] = 0.0f;
}

// Scenes with several views: one thread per primitive some view sees (the
// scene's list from preprocess, walked grid-stride), so that warps stay full
// however sparse the visibility; the other primitives keep the zeros of
// zero_scene_grads_kernel (or their sum, when accumulating).  Each lane walks
// only its own visible views (a bit mask per 32 views), so a warp runs as
// many per-view steps as its busiest lane needs.  The C = 3 instantiation
// (216 registers unbounded) is held to 128 so that four CTAs share an SM: it
// is bound by memory latency, and the occupancy outweighs its spills (the
// 16-view N=6 batch 135 -> 122 us); the C = 4 one lost time that way.
template <int C>
__global__ void __launch_bounds__(128, C == 3 ? 4 : 1) prim_backward_listed_kernel(SceneDev sc, SceneGradDev gr, ViewList vl,
                                                            const ViewDev* __restrict__ views, CfgDev cfg,
                                                            const uint32_t* __restrict__ tiles,
                                                            const float4* __restrict__ g2d,
                                                            const uint32_t* __restrict__ act_list,
                                                            const uint32_t* act_count) {
  wait_prior_grid();
  extern __shared__ ViewDev s_views[];
  for (int i = threadIdx.x; i < vl.n; i += blockDim.x) s_views[i] = views[vl.idx[i]];
  __syncthreads();
  const int64_t P = sc.P;
  const int64_t n_items = (int64_t)*act_count;
  const bool add = (cfg.flags & 4) != 0;  // add to the caller's running sum (UBS_FLAG_ACCUMULATE_GRADS)
  auto put = [&](float* dst, float v) { *dst = add ? *dst + v : v; };
  const int nr = sc.rot_mode == 0 ? 4 : 3;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_items; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = act_list[i];
    PrimIn<C> in;
    load_prim_b<C>(sc, p, in);
    PrimVI<C> vi;
    prim_stage<C>(in, sc.rot_mode, vi);
    PrimAcc<C> acc;
    acc_zero<C>(acc);
    // each lane walks only its own visible views (a bit mask per 32 views),
    // so a warp runs as many per-view steps as its busiest lane needs rather
    // than one per view that any lane sees
    for (int k0 = 0; k0 < vl.n; k0 += 32) {
      const int k1 = min(vl.n, k0 + 32);
      unsigned vis = 0;
      for (int k = k0; k < k1; ++k) vis |= (tiles[s_views[k].rec_off + (uint32_t)p] != 0 ? 1u : 0u) << (k - k0);
      while (vis) {
        const int k = k0 + __ffs(vis) - 1;
        vis &= vis - 1;
        const ViewDev& v = s_views[k];
        const uint32_t r = v.rec_off + (uint32_t)p;
        const float4 a = g2d[3 * (size_t)r], b = g2d[3 * (size_t)r + 1], c = g2d[3 * (size_t)r + 2];
        const float g[10] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y};
        prim_backward_view<C>(in, vi, v, cfg, g, acc);
      }
    }
    PrimGrad<C> out;
    prim_backward_final<C>(in, vi, sc.rot_mode, acc, out);
    for (int j = 0; j < 3; ++j) put(gr.mean_x + j * P + p, out.mx[j]);
    for (int j = 0; j < nr; ++j) put(gr.rot + j * P + p, out.rot[j]);
    for (int j = 0; j < 3; ++j) put(gr.scale_x + j * P + p, out.s[j]);
    for (int j = 0; j < 1 + C; ++j) put(gr.b + j * P + p, out.b[j]);
    put(gr.opacity + p, out.o);
    for (int j = 0; j < 3; ++j) put(gr.rgb + j * P + p, out.rgb[j]);
    if constexpr (C > 0) {
      for (int j = 0; j < C; ++j) put(gr.mean_q + j * P + p, out.mq[j]);
      for (int j = 0; j < 3 * C; ++j) put(gr.L_qx + j * P + p, out.lqx[j]);
      for (int j = 0; j < C * (C + 1) / 2; ++j) put(gr.L_q + j * P + p, out.lq[j]);
    }
  }
}

}  // namespace

cudaError_t launch_prim_backward(const SceneDev& sc, const SceneGradDev& g, const ViewList& vl, const ViewDev* views,
                                 const CfgDev& cfg, const Layout& L, char* ws, const uint32_t* act_list,
                                 const uint32_t* act_count, cudaStream_t st) {
  if (sc.P == 0) return cudaSuccess;
  const int threads = 128;
  const int64_t nblk = (sc.P + threads - 1) / threads;
  const size_t smem = sizeof(ViewDev) * vl.n;
  const uint32_t* tiles = (const uint32_t*)(ws + L.tiles);
  const float4* g2d = (const float4*)(ws + L.g2d);
  cudaError_t e = cudaSuccess;
  if (vl.n == 1 && sc.N > 3) {  // the drawn primitives of each CTA's range
    const int prims = pb_prims(sc.N, sc.P);
    const dim3 grid((unsigned)((sc.P + prims - 1) / prims));
    const uint32_t* vis = (const uint32_t*)(ws + L.vis_mask);
    switch (sc.N) {
      case 4: e = launch_dependent(prim_backward_drawn_kernel<1>, grid, dim3(kPbThreads), 0, st, sc, g, vl, views, cfg, vis, g2d, prims); break;
      case 6: e = launch_dependent(prim_backward_drawn_kernel<3>, grid, dim3(kPbThreads), 0, st, sc, g, vl, views, cfg, vis, g2d, prims); break;
      case 7: e = launch_dependent(prim_backward_drawn_kernel<4>, grid, dim3(kPbThreads), 0, st, sc, g, vl, views, cfg, vis, g2d, prims); break;
      default: return cudaErrorInvalidValue;
    }
    return e != cudaSuccess ? e : cudaGetLastError();
  }
  if (vl.n == 1) {
    e = launch_dependent(prim_backward_kernel, dim3((unsigned)nblk), dim3(threads), 0, st, sc, g, (int)vl.idx[0],
                         views, cfg, tiles, g2d);
    return e != cudaSuccess ? e : cudaGetLastError();
  }
  // several views (or none: an empty list): the listed primitives, the others
  // zeroed first unless accumulating
  if (!(cfg.flags & 4)) {
    e = launch_dependent(zero_scene_grads_kernel, dim3((unsigned)((sc.P + 255) / 256)), dim3(256), 0, st, g, sc.P,
                         sc.N - 3, sc.rot_mode == 0 ? 4 : 3);
    if (e != cudaSuccess) return e;
  }
  const unsigned blocks = (unsigned)(nblk < 152 * 8 ? nblk : 152 * 8);
  switch (sc.N) {
    case 3: e = launch_dependent(prim_backward_listed_kernel<0>, dim3(blocks), dim3(threads), smem, st, sc, g, vl, views, cfg, tiles, g2d, act_list, act_count); break;
    case 4: e = launch_dependent(prim_backward_listed_kernel<1>, dim3(blocks), dim3(threads), smem, st, sc, g, vl, views, cfg, tiles, g2d, act_list, act_count); break;
    case 6: e = launch_dependent(prim_backward_listed_kernel<3>, dim3(blocks), dim3(threads), smem, st, sc, g, vl, views, cfg, tiles, g2d, act_list, act_count); break;
    case 7: e = launch_dependent(prim_backward_listed_kernel<4>, dim3(blocks), dim3(threads), smem, st, sc, g, vl, views, cfg, tiles, g2d, act_list, act_count); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace ubs
