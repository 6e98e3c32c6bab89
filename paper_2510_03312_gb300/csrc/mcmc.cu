// mcmc.cu -- MCMC relocation of dead primitives (Sec. 4.5, primitive
// management after Deformable Beta Splatting): ubs_mcmc_relocate.
//
// A primitive is dead when its opacity is at most a threshold.  Each dead
// slot j is moved onto a live source drawn with probability proportional to
// opacity, exactly: the weight of a live primitive is the integer
// floor(o 2^24) (the float32 product is exact), the cumulative weights are
// 64-bit integers, and the source is the first primitive whose inclusive
// cumulative weight exceeds rand[j] mod (total weight).  A source drawn n
// times and its n copies take o' = 1 - (1 - o)^(1/(n+1)), which keeps their
// composited density; every other parameter of a copy is the source's, and
// the Adam moments of all touched primitives are reset.
//
// Kernels (one launch each, in order):
//   mcmc_weights_kernel  the weights' sums over chunks of 64 and blocks of 1024
//                        primitives; clears the per-primitive counts and sources
//   mcmc_scan_kernel     exclusive scan of the block sums (one block)
//   mcmc_draw_kernel     each dead slot's source, the per-source copy counts
//                        (integer atomics, exact) and the list of moved slots
//   mcmc_copy_kernel     the sources copied into the listed slots, a plane per
//                        grid row, but for the opacity
//   mcmc_touched_kernel  the touched primitives' new opacity, from the final
//                        counts, and zero moments; the caller's copy of the
//                        sources
//
// A draw is a search of the cumulative weights, bound by the latency of its
// dependent loads (a binary search in global memory took twenty); the copies
// touch 32-byte sectors for 4 bytes each, anywhere in the planes: bound by
// requests to L2, some 68 G a second here, and by address translation (a
// warp copying all planes of one slot, a page per lane, took 154 us).  So the
// copy kernel keeps each grid row in one plane and gives a listed slot to
// each lane, and the moments are zeroed in primitive order, where neighbours
// share requests.  P = 1M, K = 15, 5% dead, states larger than L2: 208 ->
// 100 us a call (draw 52 -> 20, copies and moments 151 -> 59; a thread per
// slot, most lanes idle, copied and zeroed all planes before).
#include <math.h>

#include "ubs.h"
#include "kernels.cuh"

namespace ubs {
namespace {

constexpr int kMcBlock = 1024;  // elements per scan block
constexpr int kMcChunk = 64;    // elements per chunk of the in-block search: four per lane of a half-warp
constexpr int kMcChunks = kMcBlock / kMcChunk;  // chunks per block
constexpr unsigned kMcCopyRow = 152;            // blocks per plane of the copy kernel
constexpr int kMcThreads = 256;
constexpr int kMcMaxPlanes = 64;

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct McLayout {
  size_t csum, list, boff, counts, src, header, total;
  uint32_t nb;
};

McLayout mc_layout(int64_t P) {
  McLayout L;
  L.nb = (uint32_t)((P + kMcBlock - 1) / kMcBlock);
  size_t o = 0;
  L.header = o;
  o += 256;  // total weight (u64), relocated count (i64)
  // the chunk sums (u64, 16 per block of 1024: 128 bytes a block), then the
  // list of moved slots (4 bytes each, at most P): 128 ceil(P / 1024) + 4 P
  // is at most 8 P rounded up to 256, for every P >= 1
  L.csum = o;
  L.list = o + (size_t)L.nb * kMcChunks * 8;
  o += align256((size_t)P * 8);
  L.boff = o;
  o += align256((size_t)L.nb * 8);
  L.counts = o;
  o += align256((size_t)P * 4);
  L.src = o;
  o += align256((size_t)P * 4);
  L.total = o;
  return L;
}

struct McHeader {
  unsigned long long total;
  long long relocated;
};

__device__ __forceinline__ bool is_dead(float o, float thr) { return o <= thr; }
__device__ __forceinline__ uint32_t weight_of(float o, float thr) {
  return is_dead(o, thr) ? 0u : (uint32_t)(o * 16777216.0f);  // floor for o >= 0
}

// Sum of w over the warp, exact in 64 bits.
__device__ __forceinline__ unsigned long long warp_sum_u32(uint32_t w) {
  const unsigned lo = __reduce_add_sync(0xffffffffu, w & 0xffffu), hi = __reduce_add_sync(0xffffffffu, w >> 16);
  return ((unsigned long long)hi << 16) + lo;
}

__global__ void __launch_bounds__(kMcThreads)
    mcmc_weights_kernel(const float* __restrict__ op, int64_t P, float thr, unsigned long long* __restrict__ csum,
                        unsigned long long* __restrict__ bsum, uint32_t* __restrict__ counts,
                        int32_t* __restrict__ src) {
  wait_prior_grid();
  __shared__ unsigned long long s_sum[kMcThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int E = kMcBlock / kMcThreads;  // elements per thread: two chunks per warp
  const int64_t base = (int64_t)blockIdx.x * kMcBlock + warp * (32 * E) + lane;
  float o[E];
#pragma unroll
  for (int e = 0; e < E; ++e) o[e] = base + e * 32 < P ? op[base + e * 32] : -1.0f;
  unsigned long long sum[E / 2];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int64_t i = base + e * 32;
    if (i < P) {
      counts[i] = 0;
      src[i] = -1;
    }
    const unsigned long long s = warp_sum_u32(i < P ? weight_of(o[e], thr) : 0u);
    sum[e / 2] = (e & 1) ? sum[e / 2] + s : s;
  }
  unsigned long long tot = 0;
#pragma unroll
  for (int c = 0; c < E / 2; ++c) {
    if (lane == 0) csum[(size_t)blockIdx.x * kMcChunks + warp * (E / 2) + c] = sum[c];
    tot += sum[c];
  }
  if (lane == 0) s_sum[warp] = tot;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long b = 0;
    for (int w = 0; w < kMcThreads / 32; ++w) b += s_sum[w];
    bsum[blockIdx.x] = b;
  }
}

// exclusive scan of the block sums in place (one block, sequential chunks)
__global__ void __launch_bounds__(1024) mcmc_scan_kernel(unsigned long long* __restrict__ bsum, uint32_t nb,
                                                         McHeader* hdr) {
  wait_prior_grid();
  __shared__ unsigned long long wt[32];
  __shared__ unsigned long long carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint32_t b0 = 0; b0 < nb; b0 += 1024) {
    const uint32_t i = b0 + threadIdx.x;
    const unsigned long long a = i < nb ? bsum[i] : 0ull;
    unsigned long long x = a;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) wt[warp] = x;
    __syncthreads();
    unsigned long long woff = 0;
    for (int w = 0; w < warp; ++w) woff += wt[w];
    const unsigned long long c = carry;
    if (i < nb) bsum[i] = c + woff + x - a;
    __syncthreads();
    if (threadIdx.x == 1023) carry = c + woff + x;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    hdr->total = carry;
    hdr->relocated = 0;
  }
}

struct McPlanes {
  int32_t K, op_row;
};

__device__ __forceinline__ float cloned_opacity(float o, uint32_t n) {
  return 1.0f - powf(1.0f - o, 1.0f / (float)(n + 1));
}

// inclusive sum over the lanes of a half-warp up to this one
__device__ __forceinline__ unsigned long long half_incl_scan(unsigned long long x) {
  const int lane = threadIdx.x & 15;
#pragma unroll
  for (int d = 1; d < 16; d <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, x, d, 16);
    if (lane >= d) x += y;
  }
  return x;
}

// A block draws for the dead of its `slots` slots: it lists them in shared
// memory, each thread then takes a listed slot and finds the block of
// primitives its draw falls in (every stride-th block offset is staged in
// shared memory; at most two steps' worth of offsets are then read from
// global memory for scenes of up to 4M primitives), and each half-warp
// finishes slots one after the other: the chunk sums of the block, a lane
// each, then the chunk's weights, four a lane, two dependent loads a slot.
// Where many of the slots are dead this chain is the call's time (a whole
// warp a slot, with wider scans: 1M primitives, K = 15, 95% dead 398 us, 304
// so; 20% 174, 155), so a CTA takes 1024 slots only in scenes that give two
// CTAs an SM that way, and down to 64 in smaller ones: 100K primitives, 20%
// dead 46 us with 1024, 29 with 256 (5% 32, 25); 5000, 20% 33, 20 with 64.
constexpr uint32_t kMcOffs = 1024;  // staged block offsets
inline int draw_slots(int64_t P) {
  int slots = kMcBlock;
  while (slots > 64 && (P + slots - 1) / slots < 152 * 2) slots /= 2;
  return slots;
}
__global__ void __launch_bounds__(kMcThreads)
    mcmc_draw_kernel(const float* __restrict__ op, int64_t P, float thr, const unsigned long long* __restrict__ rnd,
                     const unsigned long long* __restrict__ csum, const unsigned long long* __restrict__ boff,
                     uint32_t nb, uint32_t* __restrict__ counts, int32_t* __restrict__ src,
                     int32_t* __restrict__ list, McHeader* hdr, int slots) {
  wait_prior_grid();
  __shared__ unsigned long long s_off[kMcOffs];
  __shared__ int32_t s_slot[kMcBlock];
  __shared__ uint32_t s_n;
  __shared__ unsigned long long s_at;
  const int lane = threadIdx.x & 31;
  const unsigned long long total = hdr->total;
  if (total == 0) return;
  if (threadIdx.x == 0) s_n = 0;
  const uint32_t stride = (nb + kMcOffs - 1) / kMcOffs, n_off = (nb + stride - 1) / stride;
  for (uint32_t i = threadIdx.x; i < n_off; i += kMcThreads) s_off[i] = boff[i * stride];
  __syncthreads();
#pragma unroll
  for (int e = 0; e < kMcBlock / kMcThreads; ++e) {
    const int at_block = e * kMcThreads + threadIdx.x;
    const int64_t j = (int64_t)blockIdx.x * slots + at_block;
    const bool dead = at_block < slots && j < P && is_dead(op[j], thr);
    const unsigned all = __ballot_sync(0xffffffffu, dead);
    uint32_t at = 0;
    if (lane == 0 && all) at = atomicAdd(&s_n, (uint32_t)__popc(all));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(all & ((1u << lane) - 1u));
    if (dead) s_slot[at] = (int32_t)j;
  }
  __syncthreads();
  const uint32_t n = s_n;
  if (n == 0) return;
  if (threadIdx.x == 0) s_at = atomicAdd((unsigned long long*)&hdr->relocated, (unsigned long long)n);
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < n; i += kMcThreads) list[s_at + i] = s_slot[i];  // below P: each slot once
  // 32 slots a warp and round, spread so that few slots still use every warp
  const uint32_t n_warps = kMcThreads / 32;
  for (uint32_t w0 = threadIdx.x >> 5; w0 < n; w0 += 32 * n_warps) {
    const uint32_t i = w0 + lane * n_warps;
    const bool on = i < n;
    unsigned long long r = 0;
    uint32_t lo = 0;
    if (on) {
      r = rnd[s_slot[i]] % total;
      uint32_t hi = n_off - 1;  // the last staged offset at most r (the first, 0, is)
      while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (s_off[mid] <= r) lo = mid; else hi = mid - 1;
      }
      lo *= stride;
      hi = min(lo + stride, nb) - 1;  // then the last of the offsets up to the next staged one
      while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (boff[mid] <= r) lo = mid; else hi = mid - 1;
      }
      r -= boff[lo];
    }
    const int n_on = __popc(__ballot_sync(0xffffffffu, on));  // the first lanes
    int32_t from = -1;
    const int half = lane >> 4, sub = lane & 15;
    for (int l = 0; l < n_on; l += 2) {
      const int own = min(l + half, n_on - 1);  // this half-warp's slot
      unsigned long long rr = __shfl_sync(0xffffffffu, r, own);
      const uint32_t b = __shfl_sync(0xffffffffu, lo, own);
      // the block's first chunk whose inclusive sum exceeds rr (some chunk's does: r < total)
      const unsigned long long cs = csum[(size_t)b * kMcChunks + sub];
      unsigned long long x = half_incl_scan(cs);
      const int ch = __ffs((__ballot_sync(0xffffffffu, x > rr) >> (16 * half)) & 0xffffu) - 1;
      rr -= __shfl_sync(0xffffffffu, x - cs, ch, 16);
      // and that chunk's first primitive: four to a lane
      const int64_t p = (int64_t)b * kMcBlock + ch * kMcChunk + 4 * sub;
      unsigned long long q[4], sum = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        sum += p + k < P ? weight_of(op[p + k], thr) : 0u;
        q[k] = sum;
      }
      x = half_incl_scan(sum);
      const int f = __ffs((__ballot_sync(0xffffffffu, x > rr) >> (16 * half)) & 0xffffu) - 1;
      rr -= x - sum;  // in lane f, what is left for its four
      const int at = 4 * sub + (rr < q[0] ? 0 : rr < q[1] ? 1 : rr < q[2] ? 2 : 3);
      const int64_t g = (int64_t)b * kMcBlock + ch * kMcChunk + __shfl_sync(0xffffffffu, at, f, 16);
      const int32_t v0 = __shfl_sync(0xffffffffu, (int32_t)g, 0), v1 = __shfl_sync(0xffffffffu, (int32_t)g, 16);
      if (lane == l) from = v0;
      if (lane == l + 1) from = v1;  // n_on odd: lane l + 1 holds no slot
    }
    if (on) {
      src[s_slot[i]] = from;
      atomicAdd(&counts[from], 1u);
    }
  }
}

// Row y of the grid copies plane y of the sources into the listed slots.  A
// source is live and a slot dead, so no thread reads what another writes.  A
// slot's new opacity needs the final counts and its source's old opacity,
// which is left in the slot's raw opacity.
__global__ void __launch_bounds__(kMcThreads)
    mcmc_copy_kernel(McPlanes pl, int64_t P, float* __restrict__ act, float* __restrict__ raw,
                     const int32_t* __restrict__ src, const int32_t* __restrict__ list, const McHeader* hdr) {
  wait_prior_grid();
  const int64_t n = hdr->total ? hdr->relocated : 0;
  const size_t plane = (size_t)blockIdx.y * P;
  const bool opacity = (int)blockIdx.y == pl.op_row;
  for (int64_t i = (int64_t)blockIdx.x * kMcThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kMcThreads) {
    const int32_t j = list[i], s = src[j];
    const size_t d = plane + j, o = plane + s;
    const float a = act[o];
    if (opacity) {
      raw[d] = a;
    } else {
      act[d] = a;
      raw[d] = raw[o];
    }
  }
}

// Every touched primitive, slot or source, in its own lane: the new opacity
// (a moved slot's raw opacity holds its source's from before, a source's own
// is in place) and zero moments.  Neighbours share lines here: one request
// per warp and plane instead of one per slot and one per source.
__global__ void __launch_bounds__(kMcThreads)
    mcmc_touched_kernel(McPlanes pl, int64_t P, float* __restrict__ act, float* __restrict__ raw,
                        float* __restrict__ m, float* __restrict__ v, const uint32_t* __restrict__ counts,
                        const int32_t* __restrict__ src, int32_t* __restrict__ out, const McHeader* hdr,
                        long long* __restrict__ n_out) {
  wait_prior_grid();
  const int64_t j = (int64_t)blockIdx.x * kMcThreads + threadIdx.x;
  if (n_out && j == 0) *n_out = hdr->relocated;
  if (j >= P) return;
  const int32_t s = src[j];
  const uint32_t own = counts[j];
  if (out) out[j] = s;
  if (s < 0 && own == 0) return;
  for (int k = 0; k < pl.K; ++k) {
    m[(size_t)k * P + j] = 0.0f;
    v[(size_t)k * P + j] = 0.0f;
  }
  const size_t o = (size_t)pl.op_row * P + j;
  const float op = cloned_opacity(s >= 0 ? raw[o] : act[o], s >= 0 ? counts[s] : own);
  act[o] = op;
  raw[o] = logf(op / (1.0f - op));
}

}  // namespace
}  // namespace ubs

using namespace ubs;

extern "C" size_t ubs_mcmc_workspace_size(int64_t P) {
  if (P < 1 || P > (int64_t)0x7fffffff) return 0;
  return mc_layout(P).total;
}

extern "C" ubs_status ubs_mcmc_relocate(int32_t K, int64_t P, int32_t opacity_row, float dead_threshold,
                                        float* act, float* raw, float* m, float* v, const uint64_t* rand,
                                        int32_t* sources, int64_t* n_relocated, void* workspace,
                                        size_t workspace_bytes, cudaStream_t stream) {
  ubs::TraceRange trace_("ubs_mcmc_relocate");
  if (K < 1 || K > kMcMaxPlanes || P < 1 || P > (int64_t)0x7fffffff) return UBS_ERR_INVALID_ARG;
  if (opacity_row < 0 || opacity_row >= K || !(dead_threshold >= 0.0f && dead_threshold < 1.0f))
    return UBS_ERR_INVALID_ARG;
  if (!act || !raw || !m || !v || !rand || !workspace) return UBS_ERR_INVALID_ARG;
  if (((uintptr_t)act | (uintptr_t)raw | (uintptr_t)m | (uintptr_t)v | (uintptr_t)sources) & 3u)
    return UBS_ERR_ALIGNMENT;
  if ((((uintptr_t)rand | (uintptr_t)n_relocated) & 7u) || ((uintptr_t)workspace & 255u)) return UBS_ERR_ALIGNMENT;
  const McLayout L = mc_layout(P);
  if (workspace_bytes < L.total) return UBS_ERR_WORKSPACE;
  char* ws = (char*)workspace;
  McHeader* hdr = (McHeader*)(ws + L.header);
  unsigned long long* csum = (unsigned long long*)(ws + L.csum);
  unsigned long long* boff = (unsigned long long*)(ws + L.boff);
  uint32_t* counts = (uint32_t*)(ws + L.counts);
  int32_t* src = (int32_t*)(ws + L.src);
  int32_t* list = (int32_t*)(ws + L.list);
  const float* op = act + (size_t)opacity_row * P;
  const unsigned grid = (unsigned)((P + kMcThreads - 1) / kMcThreads);
  McPlanes pl{K, opacity_row};
  const int slots = draw_slots(P);
  cudaError_t e = launch_dependent(mcmc_weights_kernel, dim3(L.nb), dim3(kMcThreads), 0, stream, op, P,
                                   dead_threshold, csum, boff, counts, src);
  if (e == cudaSuccess) e = launch_dependent(mcmc_scan_kernel, dim3(1), dim3(1024), 0, stream, boff, L.nb, hdr);
  if (e == cudaSuccess)
    e = launch_dependent(mcmc_draw_kernel, dim3((unsigned)((P + slots - 1) / slots)), dim3(kMcThreads), 0, stream, op,
                         P, dead_threshold, (const unsigned long long*)rand, (const unsigned long long*)csum,
                         (const unsigned long long*)boff, L.nb, counts, src, list, hdr, slots);
  // a CTA a plane per 1024 slots (most hold no dead one: 100K primitives, K = 36,
  // 1% dead 27 us with one per 256, 25 so), where that leaves some for each plane
  const unsigned least = grid < 16 ? grid : 16, most = L.nb < kMcCopyRow ? L.nb : kMcCopyRow;
  const unsigned row = most < least ? least : most;
  if (e == cudaSuccess)
    e = launch_dependent(mcmc_copy_kernel, dim3(row, (unsigned)K), dim3(kMcThreads), 0, stream, pl, P, act, raw,
                         (const int32_t*)src, (const int32_t*)list, (const McHeader*)hdr);
  if (e == cudaSuccess)
    e = launch_dependent(mcmc_touched_kernel, dim3(grid), dim3(kMcThreads), 0, stream, pl, P, act, raw, m, v,
                         (const uint32_t*)counts, (const int32_t*)src, sources, (const McHeader*)hdr,
                         (long long*)n_relocated);
  return e == cudaSuccess ? UBS_OK : UBS_ERR_CUDA;
}
