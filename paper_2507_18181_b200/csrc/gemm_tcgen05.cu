// Weight-streaming projections on the 5th-generation tensor cores (sm_100a), two SMs per tile.
//
//   D[m][t] = sum_k W[m][k] * (hi[t][k] + lo[t][k])        W: [M, K] bf16, activations: two bf16 planes
//
// These kernels run a call's projections when it has more rows than the fused layer stack takes (65 to 256 tokens).
// The weight matrix is the MMA "A" operand, the tokens are the "N" dimension, and every weight byte is read from HBM
// once.  What bounds a step of this size is neither HBM nor, at first, the tensor pipe, but what has to be carried
// into shared memory: with one SM per 128-row tile the activation block of 256 tokens (64 KB per 64 columns, both
// planes) came along with every 16 KB of weights, and each N = 128 MMA fetched the weight tile again.  Hence a CTA
// pair (cta_group::2): 256 weight rows per MMA, 128 on each SM, and each SM stages only its own half of the token
// operand -- 48 instead of 80 KB per 64 columns -- in MMAs of N up to 256.
//  - Up to 128 tokens ("split planes") the two CTAs hold the two planes: the leader's half of the N dimension is the
//    hi plane, its peer's the lo plane, one MMA of N = 2 * tokens does both and the epilogue adds the halves.
//  - From 129 tokens on ("folded") each CTA holds half of the tokens in both planes; one MMA per plane, N = tokens,
//    accumulates into the same TMEM columns.  Two accumulator sets fit the 512 columns either way.
// Measured at 256 rows of the 7B shape (events around each launch): gate/up 139 -> 97 us, down 74 -> 50, QKV 33 -> 29,
// O 29 -> 25, and gate/up to 91 since (swiglu_pair); 256 rows x 4096 x 28672 in two planes is 120 GFLOP, so it runs at
// 1.32 PFLOP/s, what a cuBLAS GEMM sustains on these GPUs under their power limit (1.34; 1.63 in a burst).
//
// Scheduling.  The kernel is persistent, one CTA pair per SM pair, over (256-row tile, 64-column k-block) units.
//  - Linear outputs (QKV, O, down): the k-blocks of every tile are cut into `splits` equal parts, one pair each; it
//    writes its fp32 partial sums to plane `split` and the consumer kernel adds the planes in a fixed order.
//  - Non-linear epilogues (gate/up with SiLU * up, LM head with arg-max): the units of the whole matrix are cut
//    into equal contiguous ranges, one per pair, so every SM streams the same number of weight bytes whatever the
//    tile count.  A tile whose k-blocks fall into two ranges is summed in a fixed order: the pair holding its later
//    k-blocks (which it processes first) parks its partial sums in a workspace slot and publishes a flag; the pair
//    holding k-block 0 (which it processes last) adds them in pair order and runs the epilogue.  All pairs are
//    co-resident (the grid is what the occupancy query allows) and every flag wait is bounded.
//
// Roles: warp 0 of either CTA issues its own TMA loads (all of them complete on the leader's mbarrier), one thread of
// the leader's warp 1 issues tcgen05.mma for both, warps 2..9 of either CTA drain their own TMEM (tcgen05.ld; warps w
// and w + 4 share a lane quadrant and take alternate 16-token blocks) into the epilogue; two TMEM accumulator sets
// let the epilogue of one tile overlap the main loop of the next.
//
// Programmatic dependent launch: the weight tiles of the first pipeline stages are requested before
// the kernel waits for its predecessor in the stream, since weights never change; only activation
// loads and global writes come after that wait.
//
// Every mbarrier or flag wait is bounded by wall-clock time; on expiry the CTA records
// SPECASR_ERR_TIMEOUT in the status word, lets copies in flight land, frees its TMEM and returns.
#include "internal.h"
#include "device_utils.cuh"
#include "sm100_ptx.cuh"

using namespace sm100;

namespace {

constexpr int TILE_M = 128;           // weight rows per CTA; a pair covers two adjacent tiles
constexpr int SUB_K = 64;             // bf16 elements = 128 bytes = one swizzle row
constexpr int UMMA_K = 16;
constexpr int W_BYTES = TILE_M * SUB_K * 2;
constexpr int MAX_STAGES = 8;
constexpr int SMEM_LIMIT = 227 * 1024;  // dynamic shared memory one CTA may ask for
constexpr int EPI_TOKENS = 64;        // tokens of the SwiGLU output staged in shared memory at a time
constexpr int EPI_THREADS = 256;      // warps 2..9

struct alignas(16) SharedCtl {
  unsigned long long full[MAX_STAGES];    // the leader's are used: both CTAs' copies of a stage have landed
  unsigned long long empty[MAX_STAGES];   // each CTA's own: the MMAs have read the stage
  unsigned long long acc_full[2];         // each CTA's own
  unsigned long long acc_empty[2];        // the leader's: both CTAs' epilogues have drained the set
  unsigned long long key[SPECASR_MAX_NODES];
  uint32_t tmem_base;
  int abort;
};

struct TcParams {
  int M, n, n_pad, n_alloc, box_rows, stages, KB, tiles, ptiles, splits, epoch;
  int kt64;                 // 64-column tiles per row tile of the packed weight matrix
  int32_t* ctl;
  float* fixP;              // [grid][n_pad][128] parked partial sums (hi + lo halves added) of split tiles
  int32_t* fixFlag;         // [grid] launch number of the partial sums each CTA parked last
  float* P;                 // EPI_PARTIAL: [splits][n_alloc][M]
  bf16* A;                  // EPI_SWIGLU: [2][n_alloc][M/2]
  unsigned long long* amax; // EPI_ARGMAX: [tiles][n_alloc]
  float* logits;            // EPI_ARGMAX: optional [n][M]
#ifdef SPECASR_TRACE
  TraceBuf tr;
  int kind;                 // SPECASR_KIND_* of this launch
#endif
};

__device__ __forceinline__ int ld_acquire(const int32_t* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int32_t* p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

template <int EPI, bool FOLD>
__global__ void __launch_bounds__(64 + EPI_THREADS, 1) k_proj(const __grid_constant__ CUtensorMap tmW,
                                                 const __grid_constant__ CUtensorMap tmAct, const TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  cluster_arrive_relaxed();           // waited for below
  SPECASR_TRACE_SCOPE(p.tr, p.kind);
  uint8_t* ring = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int act_plane = p.box_rows * SUB_K * 2;           // bytes of one box of this CTA's token operand
  const int stage_bytes = W_BYTES + (FOLD ? 2 : 1) * act_plane;
  SharedCtl* sc = (SharedCtl*)(ring + (size_t)p.stages * stage_bytes);
  bf16* epi_stage = (bf16*)(sc + 1);                      // EPI_SWIGLU: [2 planes][64 tokens][64] output tile

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank();                   // 0 = leader
  const int cta = blockIdx.x, pair = cta >> 1, G = gridDim.x >> 1;
  const int KB = p.KB;
  const int U = p.ptiles * KB;
  int u0, u1;
  if (EPI == EPI_PARTIAL) {           // one tile, one part of its k-blocks
    const int tile = pair / p.splits, split = pair - tile * p.splits;
    u0 = tile * KB + split * KB / p.splits;
    u1 = tile * KB + (split + 1) * KB / p.splits;
  } else {                            // equal contiguous ranges of the whole unit list
    u0 = (int)((long long)pair * U / G);
    u1 = (int)((long long)(pair + 1) * U / G);
  }
  const int tile0 = u0 / KB, kb_first = u0 - tile0 * KB;   // the range's first unit
  const int acc_cols = (FOLD ? 1 : 2) * p.n_pad;            // TMEM columns of one accumulator set

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&sc->full[s], 1);
      mbar_init(&sc->empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sc->acc_full[b], 1);
      mbar_init(&sc->acc_empty[b], 2 * EPI_THREADS / 32);
    }
    sc->abort = 0;
    mbar_fence_init();
    tma_prefetch_desc(&tmW);
    tma_prefetch_desc(&tmAct);
  }
  __syncwarp();
  // Allocating a pair's tensor memory is one operation of both CTAs: not before the peer is known to run.  (With the
  // allocation first, now and then one CTA's went through and the other's, started a moment later, never returned; behind
  // the attention, which leaves the two SMs of a pair at different times.)
  cluster_wait();
  if (warp == 1) tmem_alloc_pair(&sc->tmem_base, 512);
  tc_fence_before();
  __syncthreads();
  cluster_sync();                     // the peer's barriers exist before anything signals them
  tc_fence_after();
  if (warp == 1) tmem_relinquish_pair();
  pdl_launch_dependents();
  const uint32_t tmem_base = sc->tmem_base;
  volatile int* abort = &sc->abort;
  int32_t* status = p.ctl + CTL_STATUS;

  if (warp == 0 && elect_one()) {
    // ---------------- TMA producer: this CTA's weight tile and its half of the token operand
    const int total = u1 - u0;
    const uint64_t once = make_evict_first();           // L2 policy of the weights
    const uint32_t full0 = map_to_cta(smem_u32(&sc->full[0]), 0);      // the leader's barriers
    int w_row = ((tile0 * 2 + rank) * p.kt64 + kb_first) * TILE_M;      // first row of the unit's packed tile
    int w_kb = kb_first;
    auto load_w = [&](int s) {                             // rows past the packed matrix arrive as zeros
      tma_load_2d_pair(ring + (size_t)s * stage_bytes, &tmW, 0, w_row, full0 + 8u * s, once);
      w_row += TILE_M;
      if (++w_kb == KB) {                                  // next tile of the pair's range
        w_kb = 0;
        w_row += (2 * p.kt64 - KB) * TILE_M;
      }
    };
    int a_kb = kb_first;
    auto load_act = [&](int s) {
      uint8_t* dst = ring + (size_t)s * stage_bytes + W_BYTES;
      if (FOLD) {
        tma_load_3d_pair(dst, &tmAct, a_kb * SUB_K, rank * p.box_rows, 0, full0 + 8u * s);
        tma_load_3d_pair(dst + act_plane, &tmAct, a_kb * SUB_K, rank * p.box_rows, 1, full0 + 8u * s);
      } else {
        tma_load_3d_pair(dst, &tmAct, a_kb * SUB_K, 0, rank, full0 + 8u * s);
      }
      if (++a_kb == KB) a_kb = 0;
    };
    // weights never change: request the first stages before waiting for the previous kernel
    const int pre = total < p.stages ? total : p.stages;
    for (int s = 0; s < pre; ++s) {
      if (rank == 0) mbar_expect_tx(&sc->full[s], (uint32_t)(2 * stage_bytes));
      load_w(s);
    }
    pdl_wait();
    SPECASR_TRACE_MARK();
    if (*(volatile int32_t*)status != 0) {
      if (pre > 0) *abort = 1;       // weight tiles are in flight: hold the shared memory until they land
    } else {
      for (int s = 0; s < pre; ++s) load_act(s);
      int s = pre == p.stages ? 0 : pre;
      uint32_t par = 0u;
      for (int i = pre; i < total; ++i) {
        if (!mbar_wait(&sc->empty[s], par, abort, status)) break;
        if (rank == 0) mbar_expect_tx(&sc->full[s], (uint32_t)(2 * stage_bytes));
        load_w(s);
        load_act(s);
        if (++s == p.stages) {
          s = 0;
          par ^= 1u;
        }
      }
      // The leader's commits arrive on both CTAs.  Those of the last stages, which nothing else waits for, have to land
      // before this CTA leaves: its shared memory then belongs to another kernel, whose barriers they would hit.
      if (total < p.stages) s = 0;
      for (int i = 0; i < pre; ++i) {
        if (!mbar_wait(&sc->empty[s], par, abort, status)) break;
        if (++s == p.stages) {
          s = 0;
          par ^= 1u;
        }
      }
    }
  } else if (warp == 1 && rank == 0 && elect_one()) {
    // ---------------- MMA issuer of the pair
    pdl_wait();
    if (*(volatile int32_t*)status == 0) {
      const uint32_t idesc = make_idesc_bf16_m256(acc_cols);
      const uint32_t ring_lo = smem_desc_lo(smem_u32(ring));
      int s = 0, kb = kb_first, b = 0;
      uint32_t par = 0u, acc_par = 1u;
      bool ok = true;
      for (int u = u0; u < u1 && ok;) {
        const int kb1 = (u1 - u) < (KB - kb) ? kb + (u1 - u) : KB;
        u += kb1 - kb;
        if (!mbar_wait(&sc->acc_empty[b], acc_par, abort, status)) break;
        tc_fence_after();
        const uint32_t d_addr = tmem_base + (uint32_t)(b * acc_cols);
        uint32_t acc = 0u;
        for (; kb < kb1; ++kb) {
          if (!mbar_wait(&sc->full[s], par, abort, status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a_lo = ring_lo + (uint32_t)((s * stage_bytes) >> 4);
          const uint32_t b_lo = a_lo + (W_BYTES >> 4);
#pragma unroll
          for (int k = 0; k < SUB_K / UMMA_K; ++k) {
            const uint32_t off = (uint32_t)((k * UMMA_K * 2) >> 4);
            umma_bf16_pair(d_addr, a_lo + off, b_lo + off, idesc, acc);
            acc = 1u;
            if (FOLD) umma_bf16_pair(d_addr, a_lo + off, b_lo + (uint32_t)(act_plane >> 4) + off, idesc, 1u);
          }
          umma_commit_pair(&sc->empty[s]);   // arrives on both CTAs once these MMAs have read the stage
          if (++s == p.stages) {
            s = 0;
            par ^= 1u;
          }
        }
        if (ok) umma_commit_pair(&sc->acc_full[b]);
        kb = 0;
        b ^= 1;
        if (b == 0) acc_par ^= 1u;
      }
    }
  } else if (warp >= 2) {
    // ---------------- epilogue: TMEM lane = output row of this CTA's tile
    pdl_wait();
    const int quad = warp & 3;
    const int row = quad * 32 + lane;
    const int etid = threadIdx.x - 64;
    const int c_first = ((warp - 2) >> 2) * 16;          // this warp's first 16-token block; the stride is 32
    bool ok = *(volatile int32_t*)status == 0;
    const uint32_t acc_empty0 = map_to_cta(smem_u32(&sc->acc_empty[0]), 0);
    int seg = 0, kb0 = kb_first, ptile = tile0;
    // value of token block [c0, c0 + 16): folded, or hi half + lo half of the accumulator
    auto load16 = [&](uint32_t lane_addr, int c0, float* v) {
      if (FOLD) {
        tmem_ld16(lane_addr + (uint32_t)c0, v);
        return;
      }
      float lo[16];
      tmem_ld16x2(lane_addr + (uint32_t)c0, lane_addr + (uint32_t)(p.n_pad + c0), v, lo);
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] += lo[j];
    };
    auto release_acc = [&](int b) {                      // this warp has read the accumulator set
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acc_empty0 + 8u * b);
    };
    for (int u = u0; u < u1; ++seg, ++ptile, kb0 = 0) {
      const int kb1 = (u1 - u) < (KB - kb0) ? kb0 + (u1 - u) : KB;
      u += kb1 - kb0;
      const int b = seg & 1;
      const int tile = ptile * 2 + rank;
      const int m = tile * TILE_M + row;
      const bool row_ok = m < p.M;
      // A pair that holds the first k-blocks of a split tile adds the partial sums parked by the pairs that hold
      // the rest.  Those were parked early in their run, so their flags are polled and the first block's parked sums
      // are requested here, while this segment's MMAs are still running.
      int last = pair;
      if (EPI != EPI_PARTIAL && kb0 == 0 && kb1 != KB)
        while (last + 1 < G && (long long)(last + 1) * U / G < (long long)(ptile + 1) * KB) ++last;
      float pk[16], pk_next[16];                          // parked sums of the next two blocks of this warp
      auto load_parked = [&](int c0, float* pk) {
#pragma unroll
        for (int j = 0; j < 16; ++j) pk[j] = 0.f;
        if (c0 < p.n_pad)
          for (int cc = pair + 1; cc <= last; ++cc) {
            const float* src = p.fixP + ((size_t)(cc * 2 + rank) * p.n_pad + c0) * TILE_M + row;
#pragma unroll
            for (int j = 0; j < 16; ++j) pk[j] += __ldcg(src + j * TILE_M);
          }
      };
      if (last > pair) {
        if (ok && etid == 0) {
          const unsigned long long t0 = global_ns();
          for (int cc = pair + 1; cc <= last && !*abort; ++cc) {
            while (ld_acquire(p.fixFlag + cc * 2 + rank) != p.epoch) {
              if (*abort) break;
              if (global_ns() - t0 > WAIT_LIMIT_NS) {
                *abort = 1;
                atomicExch(status, (int32_t)SPECASR_ERR_TIMEOUT);
                break;
              }
              __nanosleep(64);
            }
          }
        }
        epi_bar();
        if (*abort) ok = false;
        if (ok) {
          load_parked(c_first, pk);
          load_parked(c_first + 32, pk_next);
        }
      }
      if (ok) ok = mbar_wait_relaxed(&sc->acc_full[b], (uint32_t)((seg >> 1) & 1), abort, status);
      ok = __all_sync(0xFFFFFFFFu, ok ? 1 : 0) != 0;     // TMEM loads are warp-wide
      tc_fence_after();
      const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(b * acc_cols);

      if (EPI == EPI_PARTIAL) {
        if (ok) {
          float* out = p.P + (size_t)(pair % p.splits) * p.n_alloc * p.M;
          for (int c0 = c_first; c0 < p.n_pad; c0 += 32) {
            float v[16];
            load16(lane_addr, c0, v);
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (c0 + j < p.n && row_ok) out[(size_t)(c0 + j) * p.M + m] = v[j];
          }
          release_acc(b);
        }
        continue;
      }

      if (kb0 != 0) {
        // later k-blocks of a tile whose first k-blocks belong to an earlier pair: park the partial sums
        float* dst = p.fixP + (size_t)cta * p.n_pad * TILE_M;
        if (ok) {
          for (int c0 = c_first; c0 < p.n_pad; c0 += 32) {
            float v[16];
            load16(lane_addr, c0, v);
#pragma unroll
            for (int j = 0; j < 16; ++j) dst[(size_t)(c0 + j) * TILE_M + row] = v[j];
          }
          release_acc(b);
        }
        epi_bar();
        if (ok && etid == 0) st_release(p.fixFlag + cta, p.epoch);       // a release is cumulative over the barrier
        continue;
      }

      // first k-blocks of the tile (or all of them): run the epilogue on the complete sums
      if (EPI == EPI_ARGMAX) {
        for (int t = etid; t < SPECASR_MAX_NODES; t += EPI_THREADS) sc->key[t] = 0ull;
        epi_bar();
      }
      // the SwiGLU output is staged in shared memory 64 tokens at a time
      const int tok_chunk = EPI == EPI_SWIGLU && p.n_pad > EPI_TOKENS ? EPI_TOKENS : p.n_pad;
      for (int tc0 = 0; tc0 < p.n_pad; tc0 += tok_chunk) {
        if (ok) {
          const int c_end = tc0 + tok_chunk < p.n_pad ? tc0 + tok_chunk : p.n_pad;
          for (int c0 = tc0 + c_first; c0 < c_end; c0 += 32) {
            float v[16];
            load16(lane_addr, c0, v);
            if (last > pair) {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                v[j] += pk[j];
                pk[j] = pk_next[j];
              }
              load_parked(c0 + 64, pk_next);              // travels while this block and the next are worked on
            }
            if (EPI == EPI_SWIGLU) {
              // rows 2f / 2f + 1 of the tile are gate / up of feature f: the even lane of the pair finishes eight of the
              // tokens, the odd lane the other eight; both planes are staged in shared memory for 16-byte global stores
              float a[8];
              swiglu_pair(v, (lane & 1) != 0, a);
              bf16* st = epi_stage + (size_t)(c0 - tc0 + (lane & 1) * 8) * 64 + (row >> 1);
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                bf16 hi, lo;
                split_bf16(a[j], hi, lo);
                st[j * 64] = hi;
                st[EPI_TOKENS * 64 + j * 64] = lo;
              }
            } else if (EPI == EPI_ARGMAX) {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const int t = c0 + j;
                if (p.logits && t < p.n && row_ok) p.logits[(size_t)t * p.M + m] = v[j];
                // warp arg-max: largest ordered key, then the lowest row among its holders
                uint32_t key = __float_as_uint(v[j]);
                key = (key & 0x80000000u) ? ~key : (key | 0x80000000u);
                if (!row_ok) key = 0u;
                const uint32_t best = __reduce_max_sync(0xFFFFFFFFu, key);
                const uint32_t who = __reduce_min_sync(0xFFFFFFFFu, key == best ? (uint32_t)m : 0xFFFFFFFFu);
                if (lane == 0 && t < p.n && best != 0u)
                  atomicMax(&sc->key[t], ((unsigned long long)best << 32) | (unsigned long long)(0xFFFFFFFFu - who));
              }
            }
          }
        }
        if (EPI == EPI_SWIGLU) {
          epi_bar();
          if (ok) {
            const int F = p.M >> 1;
            const int f0 = tile * 64;
            int nt = p.n - tc0;                             // tokens of this chunk that exist
            nt = nt < 0 ? 0 : (nt > tok_chunk ? tok_chunk : nt);
            // 16-byte pieces of the [2][nt][64] tile: eight per token, plane by plane
            for (int idx = etid; idx < 2 * nt * 8; idx += EPI_THREADS) {
              const int plane = idx >= nt * 8 ? 1 : 0, rem = idx - plane * nt * 8;
              const int t = rem >> 3, ch = rem & 7;
              if (f0 + ch * 8 < F)
                *reinterpret_cast<uint4*>(p.A + (size_t)plane * p.n_alloc * F + (size_t)(tc0 + t) * F + f0 + ch * 8) =
                    *reinterpret_cast<const uint4*>(epi_stage + (size_t)plane * EPI_TOKENS * 64 + t * 64 + ch * 8);
            }
          }
          epi_bar();
        }
      }
      if (ok) release_acc(b);
      if (EPI == EPI_ARGMAX) {
        epi_bar();
        if (ok && tile < p.tiles)
          for (int t = etid; t < p.n; t += EPI_THREADS) p.amax[(size_t)tile * p.n_alloc + t] = sc->key[t];
        epi_bar();
      }
    }
  }

  __syncwarp();                       // one lane of warps 0 and 1 had a role: what follows is meant for whole warps
  tc_fence_before();
  __syncthreads();
  if (*abort) {
    // give copies still in flight time to land before the shared memory is handed back
    for (int i = 0; i < 64; ++i) __nanosleep(20000);
    __syncthreads();
  }
  cluster_sync();                     // neither CTA leaves while the other may still signal it or read its operands
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

template <int EPI, bool FOLD>
void launch_epi(const CUtensorMap& tmW, const CUtensorMap& tmAct, const TcParams& p, int pairs, size_t smem,
                cudaStream_t s) {
  launch_pdl_cluster(k_proj<EPI, FOLD>, dim3(2 * pairs), dim3(64 + EPI_THREADS), 2, smem, s, tmW, tmAct, p);
}

// Shape of the token operand of n_pad rows: folded or not, and the rows of one TMA box (a CTA's share of a plane).
bool tc_fold(int n_pad) { return n_pad > 128; }
int tc_box_rows(int n_pad) { return tc_fold(n_pad) ? n_pad / 2 : n_pad; }

}  // namespace

bool make_tensor_map_2d(CUtensorMap* out, const void* base, uint64_t inner, uint64_t outer, uint32_t box_inner,
                        uint32_t box_outer) {
  EncodeTiledFn enc = get_encode();
  if (!enc) {
    set_error("cuTensorMapEncodeTiled is not available from this driver");
    return false;
  }
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {inner * 2};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled failed with code %d (inner %llu, outer %llu)", (int)r,
              (unsigned long long)inner, (unsigned long long)outer);
    return false;
  }
  return true;
}

bool make_tensor_map_nd(CUtensorMap* out, const void* base, int rank, const uint64_t* dims, const uint64_t* strides,
                        const uint32_t* box) {
  EncodeTiledFn enc = get_encode();
  if (!enc) {
    set_error("cuTensorMapEncodeTiled is not available from this driver");
    return false;
  }
  cuuint64_t d[5], st[4];
  cuuint32_t b[5], es[5];
  for (int i = 0; i < rank; ++i) {
    d[i] = dims[i];
    b[i] = box[i];
    es[i] = 1;
    if (i + 1 < rank) st[i] = strides[i];
  }
  CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), d, st, b, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled (rank %d) failed with code %d", rank, (int)r);
    return false;
  }
  return true;
}

// Activation planes [2][n_alloc][K]: box = (64 columns, box_rows rows, `planes` planes).
bool make_act_map(CUtensorMap* out, const void* base, uint64_t K, uint64_t n_alloc, uint32_t box_rows, uint32_t planes) {
  EncodeTiledFn enc = get_encode();
  if (!enc) {
    set_error("cuTensorMapEncodeTiled is not available from this driver");
    return false;
  }
  cuuint64_t dims[3] = {K, n_alloc, 2};
  cuuint64_t strides[2] = {K * 2, n_alloc * K * 2};
  cuuint32_t box[3] = {64, box_rows, planes};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled (activations) failed with code %d", (int)r);
    return false;
  }
  return true;
}

int gemm_tc_tiles(int M) { return (M + TILE_M - 1) / TILE_M; }

// Rows a call's projections are padded to.  MMA N is a multiple of 16 per CTA of the pair and a folded operand is cut
// in two, so steps of 32 above 64 rows; a power of two below.
int gemm_tc_pad(int n) {
  int p = 16;
  while (p < n && p < 64) p <<= 1;
  return n <= 64 ? p : (n + 31) / 32 * 32;
}

// Index of the one-plane activation map with the box rows of n_pad (kActBoxRows lists them).
static int act_map_index(int n_pad) {
  const int rows = tc_box_rows(n_pad);
  for (int i = 0; i < kActBoxes; ++i)
    if (kActBoxRows[i] == rows) return i;
  return 0;
}

cudaError_t gemm_tc_setup(specasr_model* m) {
  cudaError_t e = cudaSuccess;
  auto raise = [&](auto kernel) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_LIMIT);
  };
  raise(k_proj<EPI_PARTIAL, false>);
  raise(k_proj<EPI_PARTIAL, true>);
  raise(k_proj<EPI_SWIGLU, false>);
  raise(k_proj<EPI_SWIGLU, true>);
  raise(k_proj<EPI_ARGMAX, false>);
  raise(k_proj<EPI_ARGMAX, true>);
  if (e != cudaSuccess) return e;
  // CTA pairs that can be resident at once: one per SM pair where the driver's partition allows it
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(m->n_sm & ~1);
  cfg.blockDim = dim3(64 + EPI_THREADS);
  cfg.dynamicSmemBytes = SMEM_LIMIT;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k_proj<EPI_SWIGLU, true>, &cfg) != cudaSuccess || n < 1) {
    cudaGetLastError();
    n = 1;
  }
  m->proj_pairs = n < m->n_sm / 2 ? n : m->n_sm / 2;
  return cudaSuccess;
}

// Number of k parts of the linear projections: tiles * parts should just fill the SM pairs.
int gemm_tc_pick_splits(const specasr_model* m, int M, int K) {
  const int ptiles = (gemm_tc_tiles(M) + 1) / 2;
  const int KB = (K + SUB_K - 1) / SUB_K;
  int s = m->proj_pairs / ptiles;
  if (s > kMaxSplitK) s = kMaxSplitK;
  if (s > KB) s = KB;
  if (s < 1) s = 1;
  return s;
}

// Bytes of the parked partial sums of a call of up to n_alloc rows, here and in the fused stack: one tile per CTA, and as much
// again (the size of a workspace is a known quantity to callers, and larger chunks have tiles of up to twice as many rows).
size_t gemm_tc_fixup_bytes(const specasr_model* m, int n_alloc) {
  return (size_t)m->n_sm * 2 * n_alloc * TILE_M * sizeof(float);
}

void launch_gemm_tc(specasr_kv* kv, const GemmArgs& a, int kind, cudaStream_t s) {
  const specasr_model* m = kv->m;
  TcParams p;
  memset(&p, 0, sizeof(p));
  p.M = a.M; p.n = a.n; p.n_pad = a.n_pad; p.n_alloc = a.n_alloc;
  p.box_rows = tc_box_rows(a.n_pad);
  const bool fold = tc_fold(a.n_pad);
  const int stage_bytes = W_BYTES + (fold ? 2 : 1) * p.box_rows * SUB_K * 2;
  const int epi_bytes = a.epilogue == EPI_SWIGLU ? 2 * EPI_TOKENS * 64 * 2 : 0;   // staged output tile
  int stages = (SMEM_LIMIT - (int)sizeof(SharedCtl) - epi_bytes - 1024) / stage_bytes;
  if (stages > MAX_STAGES) stages = MAX_STAGES;
  p.stages = stages;
  p.KB = (a.K + SUB_K - 1) / SUB_K;
  p.kt64 = packed_col_tiles(a.K);
  p.tiles = gemm_tc_tiles(a.M);
  p.ptiles = (p.tiles + 1) / 2;
  p.splits = a.epilogue == EPI_PARTIAL ? a.splits : 0;
  p.epoch = ++kv->gemm_epoch;
  p.ctl = const_cast<int32_t*>(a.ctl);
  p.fixP = kv->ws.fixP;
  p.fixFlag = kv->ws.fixFlag;
  p.P = a.P; p.A = a.A; p.amax = a.amax; p.logits = a.logits;
#ifdef SPECASR_TRACE
  p.tr = kv->trace;
  p.kind = kind;
#endif
  const int units = p.ptiles * p.KB, resident = m->proj_pairs;
  const int pairs = a.epilogue == EPI_PARTIAL ? p.ptiles * p.splits : (units < resident ? units : resident);
  const size_t smem = (size_t)stages * stage_bytes + sizeof(SharedCtl) + epi_bytes + 1024;
  const CUtensorMap& act = a.tmAct[act_map_index(a.n_pad)];
  LaunchScope scope(kv, kind, s);
  if (fold) {
    switch (a.epilogue) {
      case EPI_PARTIAL: launch_epi<EPI_PARTIAL, true>(*a.tmW, act, p, pairs, smem, s); break;
      case EPI_SWIGLU: launch_epi<EPI_SWIGLU, true>(*a.tmW, act, p, pairs, smem, s); break;
      default: launch_epi<EPI_ARGMAX, true>(*a.tmW, act, p, pairs, smem, s); break;
    }
  } else {
    switch (a.epilogue) {
      case EPI_PARTIAL: launch_epi<EPI_PARTIAL, false>(*a.tmW, act, p, pairs, smem, s); break;
      case EPI_SWIGLU: launch_epi<EPI_SWIGLU, false>(*a.tmW, act, p, pairs, smem, s); break;
      default: launch_epi<EPI_ARGMAX, false>(*a.tmW, act, p, pairs, smem, s); break;
    }
  }
}
