// preprocess.cu -- P1-P3: kernel construction, Beta-modulated conditioning
// and projection of every (view, primitive) record.
//
// Compiled with --fmad=false -prec-div=true -prec-sqrt=true -ftz=false so
// that the float32 rule set of spec32.cuh holds (see prim_forward.cuh).
//
// One launch per scene.  A primitive's view-independent part (Sigma blocks,
// Cholesky of Sigma_q, Sigma_q^{-1} Sigma_qx, beta) is built once for all the
// scene's views, so its parameters are read from HBM once per batch of views.
// Three forms (launch_preprocess): a thread per primitive that loops over the
// views (N = 3, and small scenes of one view); for one view of a larger scene
// with query dimensions, a cheap test before anything else; for several, that
// test per view and a queue of the records that pass.  Parameter planes are
// structure-of-arrays: a warp reads 32 consecutive floats per plane.
#include <atomic>

#include "kernels.cuh"
#include "prim_forward.cuh"

namespace ubs {

template <int C>
__device__ __forceinline__ void load_prim(const SceneDev& sc, int64_t p, PrimIn<C>& in) {
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

// Zeroes zero[0, n) over the grid (the binning's counters, with the first
// scene's launch).
__device__ __forceinline__ void zero_words(uint32_t* __restrict__ zero, uint32_t n) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) zero[i] = 0;
}

// The first block's part for a problem of one view (see OneView).
__device__ __forceinline__ void start_one_view(const OneView& one) {
  if (!one.on || blockIdx.x != 0) return;
  const uint32_t n = sizeof(ViewDev) / 4;
  for (uint32_t i = threadIdx.x; i < n; i += blockDim.x)
    reinterpret_cast<uint32_t*>(one.dst)[i] = reinterpret_cast<const uint32_t*>(&one.v)[i];
  for (uint32_t i = threadIdx.x; i < one.hdr_words; i += blockDim.x) one.hdr[i] = 0;
  for (int i = threadIdx.x; i < one.S; i += blockDim.x) one.act_count[i] = 0;
}

template <int C>
__global__ void __launch_bounds__(256) preprocess_kernel(SceneDev sc, ViewList vl, const ViewDev* __restrict__ views,
                                                         CfgDev cfg, float4* __restrict__ rec4,
                                                         uint32_t* __restrict__ key, uint32_t* __restrict__ tiles,
                                                         uint2* __restrict__ rect, uint32_t* __restrict__ vis_mask,
                                                         uint32_t* __restrict__ act_list, uint32_t* act_count,
                                                         uint32_t* __restrict__ zero, uint32_t nzero,
                                                         const __grid_constant__ OneView one) {
  wait_prior_grid();
  zero_words(zero, nzero);
  start_one_view(one);
  extern __shared__ ViewDev s_views[];
  if (one.on) {
    if (threadIdx.x == 0) s_views[0] = one.v;
  } else {
    for (int i = threadIdx.x; i < vl.n; i += blockDim.x) s_views[i] = views[vl.idx[i]];
  }
  __syncthreads();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= sc.P) return;
  PrimIn<C> in;
  load_prim<C>(sc, p, in);
  PrimVI<C> vi;
  prim_stage<C>(in, sc.rot_mode, vi);
  const float cr = __ldg(sc.rgb + p), cg = __ldg(sc.rgb + sc.P + p), cb = __ldg(sc.rgb + 2 * sc.P + p);
  bool any = false;  // visible in some view
  for (int k = 0; k < vl.n; ++k) {
    const ViewDev& v = s_views[k];
    ViewOut o;
    view_stage<C>(in, vi, v, cfg, o);
    any = any || o.valid;
    const uint32_t r = v.rec_off + (uint32_t)p;
    tiles[r] = o.tiles;
    {
      // the warp's 32 primitives (p aligned to 32) are one word of the
      // view's visibility mask: lane l's bit for primitive 32 (p / 32) + l
      const unsigned act = __activemask();
      const unsigned vis = __ballot_sync(act, o.valid);
      if ((threadIdx.x & 31) == (unsigned)(__ffs(act) - 1)) vis_mask[v.mask_off + (uint32_t)(p >> 5)] = vis;
    }
    if (o.valid) {
      key[r] = __float_as_uint(o.depth);
      rect[r] = make_uint2((uint32_t)o.tx0 | ((uint32_t)o.ty0 << 16), (uint32_t)o.tx1 | ((uint32_t)o.ty1 << 16));
      rec4[3 * (size_t)r + 0] = make_float4(o.mu_hi[0], o.mu_hi[1], o.mu_lo[0], o.mu_lo[1]);
      rec4[3 * (size_t)r + 1] = make_float4(o.conic[0], o.conic[1], o.conic[2], log2f(o.oq));
      rec4[3 * (size_t)r + 2] = make_float4(vi.beta_x, cr, cg, cb);
    }
  }
  // scenes with several views: the primitives some view sees, listed for the
  // parameter backward (one add per warp)
  if (vl.n > 1) {
    const unsigned act = __activemask();
    const unsigned m = __ballot_sync(act, any);
    if (m) {
      const int lane = threadIdx.x & 31, leader = __ffs(act) - 1;
      uint32_t base = 0;
      if (lane == leader) base = atomicAdd(act_count, (uint32_t)__popc(m));
      base = __shfl_sync(act, base, leader);
      if (any) act_list[base + __popc(m & ((1u << lane) - 1u))] = (uint32_t)p;
    }
  }
}

// Scenes with query dimensions (N > 3).  The query culls most records (o(q)
// below alpha_min: 6% of a 16-view N=6 batch is drawn, 2% of an N=7 one), and
// the exact conditioning costs some 300 instructions a record, most of them
// the correctly rounded divisions, square root, exp and log whose float32
// results the decisions follow.  So every (view, primitive) is first put to a
// cheap test, certain_cull, that no record the rule set draws can fail; the
// records that pass go into a per-warp queue in shared memory, and whenever 32
// are queued each lane takes one through the rule set's own conditioning,
// tests and projection, from the owner's values in shared memory.  A lane's
// arithmetic on a queued record is that of view_stage, so the outputs are the
// same bits.
// Bound by instruction issue; 16 views of 500K N=6 primitives 195 us with the
// conditioning of every record on its own lane, 152 us so; 8 views of 300K
// N=7 71 -> 53.  What is left is the view-independent stage and the queued
// records.
constexpr int kQThreads = 128, kQWarps = kQThreads / 32;
constexpr int kQCap = 64;  // queue entries per warp: 31 carried over + 32 new

// What certain_cull needs of a primitive.
template <int C>
struct CullPrim {
  float mx[3], mq[C];
  float rl[C];                 // 1 / L^_kk
  float lo[C * (C - 1) / 2 + 1];  // L^_km, m < k
  float b8[C];                 // 8 beta_qk
  float below;                 // the exponent below which o(q) is certain to fall below alpha_min
};

// Whether the record's exponent bound E_ub (see view_condition) is certain to
// lie below cull_below, from approximate y: y_k = (delta_k - sum L^_km y_m) /
// L^_kk with err_k a bound on its distance from the rule set's float32 y_k:
// the view direction's approximate normalisation and the roundings of both
// are within 2e-6 (1 + |delta_k|) and 2e-6 of each term (a dozen times the
// 1e-7 each operation can add), carried through the substitution.  The bound
// is taken at |y_k| - err_k, its negative and positive parts scaled by
// 1 -+ 1e-5, and `below` is 0.01 under cull_below, for the roundings of the
// sums.  Comparisons with NaN (a
// primitive at the camera, overflows) are false: such records are queued.
template <int C>
__device__ __forceinline__ bool certain_cull(const CullPrim<C>& p, const float (&cam)[3], float time) {
  float q[C];
  int qi = 0;
  if constexpr (C == 1 || C == 4) q[qi++] = time;
  if constexpr (C >= 3) {
    const float v0 = p.mx[0] - cam[0], v1 = p.mx[1] - cam[1], v2 = p.mx[2] - cam[2];
    float rn;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rn) : "f"(fmaf(v0, v0, fmaf(v1, v1, v2 * v2))));
    q[qi++] = v0 * rn;
    q[qi++] = v1 * rn;
    q[qi++] = v2 * rn;
  }
  float y[C], err[C], E = 0.0f;
#pragma unroll
  for (int k = 0; k < C; ++k) {
    const float d = q[k] - p.mq[k];
    float a = d, e = fmaf(2e-6f, fabsf(d), 2e-6f);
#pragma unroll
    for (int m = 0; m < k; ++m) {
      const float l = p.lo[k * (k - 1) / 2 + m];
      a = fmaf(-l, y[m], a);
      e = fmaf(fabsf(l), fmaf(2e-6f, fabsf(y[m]), err[m]), e);
    }
    y[k] = a * p.rl[k];
    err[k] = fmaf(2e-6f, fabsf(y[k]), e * p.rl[k]);
    const float ylo = fmaxf(fabsf(y[k]) - err[k], 0.0f);
    // 4 beta (ln 2 - 2 y^2), in units of 8 beta
    E = fmaf(p.b8[k], fmaf(-(1.0f - 1e-5f) * ylo, ylo, 0.5f * 0.69314718f * (1.0f + 1e-5f)), E);
  }
  return E < p.below;
}

// One view: the view-independent stage, with its 35 or so rounded divisions,
// runs once a record, and is what a culled record costs most.  The test below
// needs none of it: it forms Sigma_q and an approximate Cholesky factor and
// puts the record to the bound of certain_cull with wider error terms.  With
// every pivot at least 1/8 of its diagonal, S_kk, the errors of the rule set's
// float32 factor and of this one (rounding errors eps of S_ij <= 8 eps
// sqrt(S_ii S_jj), carried through four columns, each divided by a pivot of at
// least sqrt(S_jj / 8)) stay below 52,000 eps = 3.1e-3 of the pivot and 3000 eps
// sqrt(S_kk) of an entry, taken as kTau = 4e-3 of each; other factors are not
// judged.  Everything else is as in certain_cull; the Beta exponents' exp is
// within 1e-3 of the rule set's.
template <int C>
__device__ __forceinline__ bool certain_cull_one(const PrimIn<C>& in, float below, const float (&cam)[3], float time) {
  constexpr float kTau = 4e-3f;
  float q[C];
  int qi = 0;
  if constexpr (C == 1 || C == 4) q[qi++] = time;
  if constexpr (C >= 3) {
    const float v0 = in.mx[0] - cam[0], v1 = in.mx[1] - cam[1], v2 = in.mx[2] - cam[2];
    float rn;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rn) : "f"(fmaf(v0, v0, fmaf(v1, v1, v2 * v2))));
    q[qi++] = v0 * rn;
    q[qi++] = v1 * rn;
    q[qi++] = v2 * rn;
  }
  bool judged = true;
  float L[C * (C + 1) / 2], rl[C], y[C], err[C], E = 0.0f;
#pragma unroll
  for (int k = 0; k < C; ++k) {
    float a = q[k] - in.mq[k];
    float e = fmaf(2e-6f, fabsf(a), 2e-6f), skk = 0.0f, sd = 0.0f;
#pragma unroll
    for (int l = 0; l <= k; ++l) {
      float s = in.lqx[3 * k] * in.lqx[3 * l];
      s = fmaf(in.lqx[3 * k + 1], in.lqx[3 * l + 1], s);
      s = fmaf(in.lqx[3 * k + 2], in.lqx[3 * l + 2], s);
#pragma unroll
      for (int m = 0; m <= l; ++m) s = fmaf(in.lq[tri(k, m)], in.lq[tri(l, m)], s);
      if (l == k) skk = s;
#pragma unroll
      for (int m = 0; m < l; ++m) s = fmaf(-L[tri(k, m)], L[tri(l, m)], s);
      if (l < k) {
        L[tri(k, l)] = s * rl[l];
      } else {
        judged = judged && s >= 0.125f * skk;  // false for NaN too
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rl[k]) : "f"(s));
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(sd) : "f"(skk));
        sd *= kTau * 1.01f;
      }
    }
#pragma unroll
    for (int m = 0; m < k; ++m) {
      a = fmaf(-L[tri(k, m)], y[m], a);
      e = fmaf(fabsf(L[tri(k, m)]) + sd, err[m], fmaf(sd, fabsf(y[m]), e));
    }
    y[k] = a * rl[k];
    err[k] = fmaf(kTau, fabsf(y[k]), 1.01f * e * rl[k]);
    const float ylo = fmaxf(fabsf(y[k]) - err[k], 0.0f);
    const float b8 = 8.0f * __expf(in.b[1 + k]);
    E = fmaf(b8, fmaf(-(1.0f - 1e-3f) * ylo, ylo, 0.5f * 0.69314718f * (1.0f + 1e-3f)), E);
  }
  return judged && E < below;
}

// A CTA's kOnePrims primitives: first each thread tests its own, and lists the
// ones not culled in shared memory; then the listed ones go through the rule
// set, one a thread, their parameters read again (in L1 and L2).
// 300K N=7 primitives, 1.4% drawn: 31 us with every one through the rule set,
// 17.6 us so; 200K N=6, 7% drawn: 22 -> 14.6.  Held to 64 registers, four CTAs
// an SM, with spills: against three at 80 the forward of one view is 1-3%
// slower at 200K primitives, 3-10% faster at 300K, which are one wave of CTAs
// only so, and from 600K to 2M 0-5% faster for N = 4 and 6 and equal for N = 7,
// whether the query culls most or few.
constexpr int kOneThreads = 256, kOnePrims = 512;
// Below kOneMin primitives preprocess_kernel takes the scene, in CTAs of
// kFewThreads: its grid then fills the GPU where that of kOnePrims a CTA does
// not, and there is no second read.  Forward of one 640x360 view, that / this
// form, us: 20K N=7 31 / 35 where the query culls almost all and 50 / 61 where
// it culls none; 80K 37 / 38 and 104 / 116; 100K 41 / 39 and 125 / 134; 300K
// 62 / 50 and 201 / 207.  From the line on the test pays where the query culls
// and costs at most 7% where it does not.
constexpr int64_t kOneMin = 100000;
constexpr int kFewThreads = 64;
template <int C>
__global__ void __launch_bounds__(kOneThreads, 4) preprocess_one_view_kernel(
    SceneDev sc, ViewList vl, const ViewDev* __restrict__ views, CfgDev cfg, float4* __restrict__ rec4,
    uint32_t* __restrict__ key, uint32_t* __restrict__ tiles, uint2* __restrict__ rect,
    uint32_t* __restrict__ vis_mask, uint32_t* __restrict__ zero, uint32_t nzero,
    const __grid_constant__ OneView one) {
  wait_prior_grid();
  zero_words(zero, nzero);
  start_one_view(one);
  __shared__ ViewDev s_view;
  __shared__ uint32_t s_vis[kOnePrims / 32], s_n;
  __shared__ uint16_t s_list[kOnePrims];
  if (threadIdx.x < sizeof(ViewDev) / 4)
    reinterpret_cast<uint32_t*>(&s_view)[threadIdx.x] =
        one.on ? reinterpret_cast<const uint32_t*>(&one.v)[threadIdx.x]
               : reinterpret_cast<const uint32_t*>(views + vl.idx[0])[threadIdx.x];
  if (threadIdx.x < kOnePrims / 32) s_vis[threadIdx.x] = 0;
  if (threadIdx.x == 0) s_n = 0;
  __syncthreads();
  const ViewDev& v = s_view;
  const int64_t p0 = (int64_t)blockIdx.x * kOnePrims;
  const unsigned lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < kOnePrims; i += kOneThreads) {
    const int64_t p = p0 + i + threadIdx.x, P = sc.P;
    bool cand = false;
    if (p < P) {
      PrimIn<C> in;  // what the test reads
      for (int j = 0; j < 3; ++j) in.mx[j] = __ldg(sc.mean_x + j * P + p);
      for (int j = 0; j < C; ++j) in.mq[j] = __ldg(sc.mean_q + j * P + p);
      for (int j = 0; j < C; ++j) in.b[1 + j] = __ldg(sc.b + (1 + j) * P + p);
      for (int j = 0; j < 3 * C; ++j) in.lqx[j] = __ldg(sc.L_qx + j * P + p);
      for (int j = 0; j < C * (C + 1) / 2; ++j) in.lq[j] = __ldg(sc.L_q + j * P + p);
      const float o = __ldg(sc.opacity + p);
      float cam[3];  // the camera's centre, as view_condition forms it
      for (int j = 0; j < 3; ++j) cam[j] = -((v.R[j] * v.t[0] + v.R[3 + j] * v.t[1]) + v.R[6 + j] * v.t[2]);
      const float below = cfg.amin > 0.0f ? __logf(__fdividef(cfg.amin, o)) - 0.02f : -INFINITY;
      cand = !certain_cull_one<C>(in, below, cam, v.time);
      if (!cand) tiles[v.rec_off + (uint32_t)p] = 0;
    }
    const unsigned m = __ballot_sync(0xffffffffu, cand);
    uint32_t base = 0;
    if (lane == 0 && m) base = atomicAdd(&s_n, (uint32_t)__popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (cand) s_list[base + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(i + threadIdx.x);
  }
  __syncthreads();
  const uint32_t n = s_n;
  for (uint32_t j = threadIdx.x; j < n; j += kOneThreads) {
    const uint32_t l = s_list[j];
    const int64_t p = p0 + l;
    const uint32_t r = v.rec_off + (uint32_t)p;
    PrimIn<C> in;
    PrimVI<C> vi;
    load_prim<C>(sc, p, in);
    prim_stage<C>(in, sc.rot_mode, vi);
    ViewOut o;
    view_stage<C>(in, vi, v, cfg, o);
    tiles[r] = o.tiles;
    if (o.valid) {
      atomicOr(&s_vis[l >> 5], 1u << (l & 31));
      key[r] = __float_as_uint(o.depth);
      rect[r] = make_uint2((uint32_t)o.tx0 | ((uint32_t)o.ty0 << 16), (uint32_t)o.tx1 | ((uint32_t)o.ty1 << 16));
      rec4[3 * (size_t)r + 0] = make_float4(o.mu_hi[0], o.mu_hi[1], o.mu_lo[0], o.mu_lo[1]);
      rec4[3 * (size_t)r + 1] = make_float4(o.conic[0], o.conic[1], o.conic[2], log2f(o.oq));
      rec4[3 * (size_t)r + 2] = make_float4(vi.beta_x, __ldg(sc.rgb + p), __ldg(sc.rgb + sc.P + p),
                                            __ldg(sc.rgb + 2 * sc.P + p));
    }
  }
  __syncthreads();
  if (threadIdx.x < kOnePrims / 32 && p0 + 32 * (int64_t)threadIdx.x < sc.P)
    vis_mask[v.mask_off + (uint32_t)(p0 >> 5) + threadIdx.x] = s_vis[threadIdx.x];
}

// The queued record's primitive: the fields of PrimIn and PrimVI that the
// conditioning and the projection read, a float per lane each.
template <int C>
struct QFields {
  static constexpr int kMx = 0, kMq = 3, kLh = kMq + C, kW3 = kLh + C * (C + 1) / 2, kBq = kW3 + 3 * C, kO = kBq + C,
                       kSc = kO + 1, kBx = kSc + 6, kRgb = kBx + 1, kBelow = kRgb + 3, kN = kBelow + 1;
};

template <int C>
__global__ void __launch_bounds__(kQThreads, 6) preprocess_queued_kernel(
    SceneDev sc, ViewList vl, const ViewDev* __restrict__ views, CfgDev cfg, float4* __restrict__ rec4,
    uint32_t* __restrict__ key, uint32_t* __restrict__ tiles, uint2* __restrict__ rect,
    uint32_t* __restrict__ vis_mask, uint32_t* __restrict__ act_list, uint32_t* act_count,
    uint32_t* __restrict__ zero, uint32_t nzero) {
  wait_prior_grid();
  zero_words(zero, nzero);
  using F = QFields<C>;
  extern __shared__ ViewDev s_views[];
  __shared__ float s_prim[kQWarps][F::kN][32];
  __shared__ uint32_t s_q[kQWarps][kQCap];         // view | owner lane << 16
  __shared__ uint32_t s_any[kQWarps];
  __shared__ uint32_t s_vis[kQWarps][kMaxViews];   // per warp and view: the visibility mask word
  for (int i = threadIdx.x; i < vl.n; i += kQThreads) s_views[i] = views[vl.idx[i]];
  if (threadIdx.x < kQWarps) s_any[threadIdx.x] = 0;
  for (int i = threadIdx.x; i < kQWarps * vl.n; i += kQThreads) s_vis[i / vl.n][i % vl.n] = 0;
  __syncthreads();
  const int64_t p = (int64_t)blockIdx.x * kQThreads + threadIdx.x;
  const bool live = p < sc.P;  // every lane stays: the queue is warp-synchronous
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t p0 = (uint32_t)(p - lane);  // the warp's first primitive (P is below 2^31)
  const unsigned lt = (1u << lane) - 1u;
  float(*prim)[32] = s_prim[w];
  uint32_t* queue = s_q[w];
  CullPrim<C> cp;
  cp.below = -INFINITY;  // no certain cull
  if (live) {
    PrimIn<C> in;
    PrimVI<C> vi;
    load_prim<C>(sc, p, in);
    prim_stage<C>(in, sc.rot_mode, vi);
    // the log-opacity bound below which a record is certainly culled (see
    // view_condition): approximate log and quotient, inside the bound's margin
    float cull_below = -INFINITY;
    if (cfg.amin > 0.0f) cull_below = __logf(__fdividef(cfg.amin, in.o)) - 0.01f;
    if (!vi.valid) cull_below = INFINITY;  // a record of an invalid kernel is never drawn
    for (int i = 0; i < 3; ++i) cp.mx[i] = in.mx[i];
    for (int k = 0; k < C; ++k) {
      cp.mq[k] = in.mq[k];
      cp.rl[k] = __frcp_rn(vi.Lh[tri(k, k)]);
      cp.b8[k] = 8.0f * vi.beta_q[k];
      for (int m = 0; m < k; ++m) cp.lo[k * (k - 1) / 2 + m] = vi.Lh[tri(k, m)];
    }
    cp.below = cull_below - 0.01f;
    for (int i = 0; i < 3; ++i) prim[F::kMx + i][lane] = in.mx[i];
    for (int i = 0; i < C; ++i) prim[F::kMq + i][lane] = in.mq[i];
    for (int i = 0; i < C * (C + 1) / 2; ++i) prim[F::kLh + i][lane] = vi.Lh[i];
    for (int i = 0; i < 3; ++i)
      for (int k = 0; k < C; ++k) prim[F::kW3 + i * C + k][lane] = vi.W3[i][k];
    for (int i = 0; i < C; ++i) prim[F::kBq + i][lane] = vi.beta_q[i];
    prim[F::kO][lane] = in.o;
    for (int i = 0; i < 6; ++i) prim[F::kSc + i][lane] = vi.Sc[i];
    prim[F::kBx][lane] = vi.beta_x;
    for (int i = 0; i < 3; ++i) prim[F::kRgb + i][lane] = __ldg(sc.rgb + i * sc.P + p);
    prim[F::kBelow][lane] = cull_below;
  }
  __syncwarp();
  // queue entry j through the rule set (any lane may take any entry)
  auto take = [&](int j) {
    const uint32_t e = queue[j];
    const int k = (int)(e & 0xffffu), owner = (int)(e >> 16);
    const ViewDev& v = s_views[k];
    const uint32_t r = v.rec_off + p0 + (uint32_t)owner;
    PrimIn<C> in;
    PrimVI<C> vi;
    for (int i = 0; i < 3; ++i) in.mx[i] = prim[F::kMx + i][owner];
    for (int i = 0; i < C; ++i) in.mq[i] = prim[F::kMq + i][owner];
    for (int i = 0; i < C * (C + 1) / 2; ++i) vi.Lh[i] = prim[F::kLh + i][owner];
    for (int i = 0; i < 3; ++i)
      for (int m = 0; m < C; ++m) vi.W3[i][m] = prim[F::kW3 + i * C + m][owner];
    for (int i = 0; i < C; ++i) vi.beta_q[i] = prim[F::kBq + i][owner];
    in.o = prim[F::kO][owner];
    ViewCond c;
    view_condition<C>(in, vi, v, c, prim[F::kBelow][owner]);
    // an invalid kernel's bound is infinite (as is that of an opacity of zero, and
    // one below zero has none: neither reaches alpha_min)
    if (!view_candidate(prim[F::kBelow][owner] < INFINITY, c, v, cfg)) {
      tiles[r] = 0;
      return;
    }
    float Sc[6];
    for (int i = 0; i < 6; ++i) Sc[i] = prim[F::kSc + i][owner];
    const float beta_x = prim[F::kBx][owner];
    ViewOut o;
    view_project(in.mx, Sc, beta_x, true, c, v, cfg, o);
    tiles[r] = o.tiles;
    if (o.valid) {
      atomicOr(&s_vis[w][k], 1u << owner);
      key[r] = __float_as_uint(o.depth);
      rect[r] = make_uint2((uint32_t)o.tx0 | ((uint32_t)o.ty0 << 16), (uint32_t)o.tx1 | ((uint32_t)o.ty1 << 16));
      rec4[3 * (size_t)r + 0] = make_float4(o.mu_hi[0], o.mu_hi[1], o.mu_lo[0], o.mu_lo[1]);
      rec4[3 * (size_t)r + 1] = make_float4(o.conic[0], o.conic[1], o.conic[2], log2f(o.oq));
      rec4[3 * (size_t)r + 2] =
          make_float4(beta_x, prim[F::kRgb][owner], prim[F::kRgb + 1][owner], prim[F::kRgb + 2][owner]);
      atomicOr(&s_any[w], 1u << owner);
    }
  };
  int qn = 0;  // warp-uniform
  for (int k = 0; k <= vl.n; ++k) {
    if (k < vl.n) {
      const ViewDev& v = s_views[k];
      bool cand = false;
      if (live) {
        float cam[3];  // the camera's centre, as view_condition forms it
        for (int i = 0; i < 3; ++i) cam[i] = -((v.R[i] * v.t[0] + v.R[3 + i] * v.t[1]) + v.R[6 + i] * v.t[2]);
        cand = !certain_cull<C>(cp, cam, v.time);
        if (!cand) tiles[v.rec_off + (uint32_t)p] = 0;
      }
      const unsigned m = __ballot_sync(0xffffffffu, cand);
      if (cand) queue[qn + __popc(m & lt)] = (uint32_t)k | ((uint32_t)lane << 16);
      qn += __popc(m);
      __syncwarp();
    }
    // the 32 newest entries, one per lane; after the last view, the rest
    if (qn >= 32 || (k == vl.n && qn > 0)) {
      const int n = min(qn, 32);
      if (lane < n) take(qn - n + lane);
      qn -= n;
      __syncwarp();
    }
  }
  __syncwarp();
  // the warp's visibility mask word of each view (its primitives start at a
  // multiple of 32)
  if ((int64_t)p0 < sc.P)
    for (int k = lane; k < vl.n; k += 32) vis_mask[s_views[k].mask_off + (p0 >> 5)] = s_vis[w][k];
  // scenes with several views: the primitives some view sees, listed for the
  // parameter backward (one add per warp)
  const bool any = live && ((s_any[w] >> lane) & 1u);
  if (vl.n > 1) {
    const unsigned m = __ballot_sync(0xffffffffu, any);
    if (m) {
      uint32_t base = 0;
      if (lane == 0) base = atomicAdd(act_count, (uint32_t)__popc(m));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (any) act_list[base + __popc(m & lt)] = (uint32_t)p;
    }
  }
}

constexpr int kMaxDevices = 64;
std::atomic<bool> g_queued_smem_set[kMaxDevices];

// the queued kernels' view table plus their static queues can pass 48 KB of
// shared memory (256 views): opt in once per device
cudaError_t prepare_queued() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < kMaxDevices && g_queued_smem_set[dev].load(std::memory_order_acquire)) return cudaSuccess;
  const int bytes = (int)(kMaxViews * sizeof(ViewDev));
  e = cudaFuncSetAttribute(preprocess_queued_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(preprocess_queued_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(preprocess_queued_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && dev >= 0 && dev < kMaxDevices) g_queued_smem_set[dev].store(true, std::memory_order_release);
  return e;
}

cudaError_t launch_preprocess(const SceneDev& sc, const ViewList& vl, const ViewDev* views, const CfgDev& cfg,
                              const Layout& L, char* ws, uint32_t* act_list, uint32_t* act_count, uint32_t* zero,
                              uint32_t nzero, const OneView& one, cudaStream_t st) {
  if (sc.P == 0 || vl.n == 0) return cudaSuccess;
  float4* rec4 = (float4*)(ws + L.rec4);
  uint32_t* key = (uint32_t*)(ws + L.key);
  uint32_t* tiles = (uint32_t*)(ws + L.tiles);
  uint2* rect = (uint2*)(ws + L.rect);
  uint32_t* vis = (uint32_t*)(ws + L.vis_mask);
  const size_t smem = sizeof(ViewDev) * vl.n;
  if (sc.N > 3 && vl.n == 1) {
    if (sc.P < kOneMin) {
      const dim3 grid((unsigned)((sc.P + kFewThreads - 1) / kFewThreads)), block(kFewThreads);
      switch (sc.N) {
        case 4: launch_dependent(preprocess_kernel<1>, grid, block, smem, st, sc, vl, views, cfg, rec4, key, tiles, rect, vis, act_list, act_count, zero, nzero, one); break;
        case 6: launch_dependent(preprocess_kernel<3>, grid, block, smem, st, sc, vl, views, cfg, rec4, key, tiles, rect, vis, act_list, act_count, zero, nzero, one); break;
        case 7: launch_dependent(preprocess_kernel<4>, grid, block, smem, st, sc, vl, views, cfg, rec4, key, tiles, rect, vis, act_list, act_count, zero, nzero, one); break;
        default: return cudaErrorInvalidValue;
      }
      return cudaGetLastError();
    }
    const dim3 grid((unsigned)((sc.P + kOnePrims - 1) / kOnePrims)), block(kOneThreads);
    switch (sc.N) {
      case 4: launch_dependent(preprocess_one_view_kernel<1>, grid, block, 0, st, sc, vl, views, cfg, rec4, key, tiles, rect, vis, zero, nzero, one); break;
      case 6: launch_dependent(preprocess_one_view_kernel<3>, grid, block, 0, st, sc, vl, views, cfg, rec4, key, tiles, rect, vis, zero, nzero, one); break;
      case 7: launch_dependent(preprocess_one_view_kernel<4>, grid, block, 0, st, sc, vl, views, cfg, rec4, key, tiles, rect, vis, zero, nzero, one); break;
      default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
  }
  if (sc.N > 3) {
    const cudaError_t e = prepare_queued();
    if (e != cudaSuccess) return e;
  }
  const int threads = sc.N > 3 ? kQThreads : 256;
  const unsigned blocks = (unsigned)((sc.P + threads - 1) / threads);
  switch (sc.N) {
    case 3: launch_dependent(preprocess_kernel<0>, dim3(blocks), dim3(threads), smem, st, sc, vl, views, cfg, rec4, key, tiles, rect, vis, act_list, act_count, zero, nzero, one); break;
    case 4: launch_dependent(preprocess_queued_kernel<1>, dim3(blocks), dim3(threads), smem, st, sc, vl, views, cfg, rec4, key, tiles, rect, vis, act_list, act_count, zero, nzero); break;
    case 6: launch_dependent(preprocess_queued_kernel<3>, dim3(blocks), dim3(threads), smem, st, sc, vl, views, cfg, rec4, key, tiles, rect, vis, act_list, act_count, zero, nzero); break;
    case 7: launch_dependent(preprocess_queued_kernel<4>, dim3(blocks), dim3(threads), smem, st, sc, vl, views, cfg, rec4, key, tiles, rect, vis, act_list, act_count, zero, nzero); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace ubs
