// specasr_top2_probs: the two most probable tokens of every row of a logits matrix and their softmax
// probabilities over the whole vocabulary -- the quantities the draft side of the method reads (Section IV-A:
// drafting stops where the normalised top-1 value falls below a threshold; Section IV-C: the second-ranked
// token at such a position seeds a side branch).  See include/specasr.h for the contract.
//
// One to eight CTAs (a cluster) per row.  Every thread scans a strided part of its CTA's slice once, keeping its two largest
// packed (ordered logit, ~token id) keys and an online (max, sum of exp) pair; warps, CTAs and the cluster merge those.
#include <cooperative_groups.h>

#include "internal.h"
#include "device_utils.cuh"

namespace {

struct Top2 {
  unsigned long long a, b;     // a >= b, 0 = empty
};
__device__ __forceinline__ void top2_push(Top2& t, unsigned long long k) {
  if (k > t.a) {
    t.b = t.a;
    t.a = k;
  } else if (k > t.b) {
    t.b = k;
  }
}
__device__ __forceinline__ float key_value(unsigned long long k) {
  uint32_t u = (uint32_t)(k >> 32);
  u = (u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u;
  return __uint_as_float(u);
}
// (m, s) with s = sum of exp(x - m) over the elements seen so far; m = -inf and s = 0 when none but -inf
__device__ __forceinline__ void lse_merge(float& m, float& s, float m2, float s2) {
  const float mm = fmaxf(m, m2);
  const float ref = mm > -INFINITY ? mm : 0.f;      // nothing to subtract while both have seen nothing
  s = s * expf(m - ref) + s2 * expf(m2 - ref);
  m = mm;
}

// One cluster of CTAs per row: each takes a slice of the vocabulary, the partial results meet in the first CTA's shared
// memory and are merged in slice order.  Bound by the latency of a slice, not by bandwidth: with one block per row each
// thread ran through 125 dependent (max, sum) updates of a 32000-token row; a thread now loads eight values at a time,
// takes their maximum first, and a row is spread over up to eight SMs.
constexpr int kTop2Cluster = 8;          // CTAs per row, at most
struct Top2Part {
  Top2 t;
  float m, s;
};
__device__ __forceinline__ void top2_merge(Top2Part& a, const Top2Part& b) {
  top2_push(a.t, b.t.a);
  top2_push(a.t, b.t.b);
  lse_merge(a.m, a.s, b.m, b.s);
}
__global__ void __launch_bounds__(256) k_top2_probs(const float* __restrict__ logits, int vocab,
                                                    int32_t* __restrict__ out_ids, float* __restrict__ out_probs) {
  namespace cg = cooperative_groups;
  __shared__ Top2Part s_warp[8];
  __shared__ Top2Part s_part[kTop2Cluster];
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), parts = (int)cluster.num_blocks();
  const int row_id = blockIdx.x / parts;
  cluster.barrier_arrive();                  // waited for before the first write into another CTA: it has started
  grid_dep_launch();
  grid_dep_wait();
  // indices count from the slice's start: what a thread reads ahead of a row's end would pass 2^31 in the widest vocabularies
  const int v0 = (int)((long long)rank * vocab / parts), len = (int)((long long)(rank + 1) * vocab / parts) - v0;
  const float* slice = logits + (size_t)row_id * vocab + v0;
  Top2Part p{{0ull, 0ull}, -INFINITY, 0.f};
  for (int base = threadIdx.x; base < len; base += 256 * 8) {
    float x[8];
    float top = p.m;
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = base + u * 256 < len ? slice[base + u * 256] : -INFINITY;
#pragma unroll
    for (int u = 0; u < 8; ++u) top = fmaxf(top, x[u]);
    // masked values (-inf) count for nothing; while a thread has seen nothing else there is no maximum to subtract
    const float ref = top > -INFINITY ? top : 0.f;
    p.s *= expf(p.m - ref);                 // expf(-inf) = 0 covers the first values
    p.m = top;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (base + u * 256 < len) {
        p.s += expf(x[u] - ref);
        top2_push(p.t, pack_max_key(x[u], (uint32_t)(v0 + base + u * 256)));
      }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Top2Part q;
    q.t.a = __shfl_xor_sync(0xFFFFFFFFu, p.t.a, o);
    q.t.b = __shfl_xor_sync(0xFFFFFFFFu, p.t.b, o);
    q.m = __shfl_xor_sync(0xFFFFFFFFu, p.m, o);
    q.s = __shfl_xor_sync(0xFFFFFFFFu, p.s, o);
    top2_merge(p, q);
  }
  if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = p;
  __syncthreads();
  cluster.barrier_wait();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) top2_merge(p, s_warp[w]);
    *cluster.map_shared_rank(&s_part[rank], 0) = p;
  }
  cluster.sync();                            // afterwards only the first CTA reads, and only its own shared memory
  if (rank == 0 && threadIdx.x == 0) {
    p = s_part[0];
    for (int q = 1; q < parts; ++q) top2_merge(p, s_part[q]);
    Top2& t = p.t;
    if (t.b == 0ull) t.b = t.a;                    // a one-token vocabulary
    int32_t* ids = out_ids + (size_t)row_id * 2;
    float* pr = out_probs + (size_t)row_id * 2;
    ids[0] = (int32_t)(0xFFFFFFFFu - (uint32_t)(t.a & 0xFFFFFFFFull));
    ids[1] = (int32_t)(0xFFFFFFFFu - (uint32_t)(t.b & 0xFFFFFFFFull));
    pr[0] = expf(key_value(t.a) - p.m) / p.s;
    pr[1] = expf(key_value(t.b) - p.m) / p.s;
  }
}

// The same two tokens and probabilities from what the vocabulary projection's epilogue left per 128-row tile
// (best and second-best packed key, max and sum of exp): one block per node, threads stride over the tiles.
__global__ void __launch_bounds__(256) k_top2_from_tiles(const __grid_constant__ SegTable tab,
                                                         const int32_t* __restrict__ ctl_shared,
                                                         const unsigned long long* __restrict__ first,
                                                         const unsigned long long* __restrict__ second,
                                                         const float2* __restrict__ lse, int n_tiles, int n_alloc,
                                                         int32_t* __restrict__ out_ids, float* __restrict__ out_probs) {
  __shared__ Top2 s_top[8];
  __shared__ float s_m[8], s_s[8];
  grid_dep_launch();
  grid_dep_wait();
  const int node = blockIdx.x;
  int b = 0;
  while (b + 1 < tab.count && node >= tab.seg[b].row0 + tab.seg[b].n) ++b;
  int32_t* ids = out_ids + (size_t)node * 2;
  float* pr = out_probs + (size_t)node * 2;
  if (tab.seg[b].ctl[CTL_STATUS] != 0 || (ctl_shared && ctl_shared[CTL_STATUS] != 0)) {
    if (threadIdx.x == 0) {
      ids[0] = ids[1] = -1;
      pr[0] = pr[1] = 0.f;
    }
    return;
  }
  Top2 t{0ull, 0ull};
  float m = -INFINITY, s = 0.f;
  for (int tile = threadIdx.x; tile < n_tiles; tile += 256) {
    top2_push(t, __ldcg(first + (size_t)tile * n_alloc + node));
    top2_push(t, __ldcg(second + (size_t)tile * n_alloc + node));
    const float2 ms = __ldcg(lse + (size_t)tile * n_alloc + node);
    lse_merge(m, s, ms.x, ms.y);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long oa = __shfl_xor_sync(0xFFFFFFFFu, t.a, o), ob = __shfl_xor_sync(0xFFFFFFFFu, t.b, o);
    top2_push(t, oa);
    top2_push(t, ob);
    const float om = __shfl_xor_sync(0xFFFFFFFFu, m, o), os = __shfl_xor_sync(0xFFFFFFFFu, s, o);
    lse_merge(m, s, om, os);
  }
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    s_top[warp] = t;
    s_m[warp] = m;
    s_s[warp] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) {
      top2_push(t, s_top[w].a);
      top2_push(t, s_top[w].b);
      lse_merge(m, s, s_m[w], s_s[w]);
    }
    if (t.b == 0ull) t.b = t.a;                    // a one-token vocabulary
    ids[0] = (int32_t)(0xFFFFFFFFu - (uint32_t)(t.a & 0xFFFFFFFFull));
    ids[1] = (int32_t)(0xFFFFFFFFu - (uint32_t)(t.b & 0xFFFFFFFFull));
    pr[0] = expf(key_value(t.a) - m) / s;
    pr[1] = expf(key_value(t.b) - m) / s;
  }
}

}  // namespace

void launch_top2_from_tiles(specasr_kv* wk, const SegTable& t, const int32_t* ctl_shared, int n_total, int n_tiles,
                            int32_t* out_ids, float* out_probs, cudaStream_t s) {
  LaunchScope scope(wk, SPECASR_KIND_ACCEPT, s);
  launch_pdl(k_top2_from_tiles, dim3(n_total), dim3(256), 0, s, t, ctl_shared, wk->ws.amax, wk->ws.sec, wk->ws.lse, n_tiles,
             wk->n_alloc, out_ids, out_probs);
}

extern "C" specasr_status specasr_top2_probs(const float* logits, int32_t n_rows, int32_t vocab, int32_t* out_ids,
                                             float* out_probs, void* stream) {
  if (!logits || !out_ids || !out_probs) {
    set_error("specasr_top2_probs: null argument");
    return SPECASR_ERR_INVALID_ARG;
  }
  if (n_rows < 1 || vocab < 1) {
    set_error("specasr_top2_probs: n_rows = %d and vocab = %d must be positive", n_rows, vocab);
    return SPECASR_ERR_INVALID_ARG;
  }
  int parts = 1;                               // CTAs per row: at least eight values per thread
  while (parts < kTop2Cluster && vocab / (2 * parts) >= 2048) parts *= 2;
  launch_pdl_cluster(k_top2_probs, dim3(parts * n_rows), dim3(256), parts, 0, (cudaStream_t)stream, logits, vocab, out_ids,
                     out_probs);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("specasr_top2_probs: %s", cudaGetErrorString(e));
    return SPECASR_ERR_CUDA;
  }
  return SPECASR_OK;
}
