// Tree-masked grouped-query attention as a kernel of its own (calls of more rows than the fused layer stack takes), and
// the plan of attention units that both paths follow.  What a unit does is in attention_unit.cuh.
//
// One CTA per SM walks the units u, u + grid, ...; warp 0 is the TMA producer, one thread of warp 1 issues the MMAs,
// warps 2..9 run the soft-max and the output.  The roles run ahead of one another from unit to unit.
//
// Every mbarrier wait is bounded; on expiry the CTA records SPECASR_ERR_TIMEOUT, lets copies in
// flight land, frees its TMEM and returns.
#include "attention_unit.cuh"

using namespace sm100;

namespace {

constexpr int ATTN_THREADS = 64 + 256;

struct AttnCtl {
  attn::Ctl a;
  uint32_t tmem_base;
  int abort;
};

struct AttnParams {
  const unsigned long long* anc;
  float* attO;
  float2* attML;
  size_t rows_alloc;      // rows of one key range's partials
  int page_size, layer, Hq, Hkv, group, nodes_per_tile;
  float scale_log2;
#ifdef SPECASR_TRACE
  TraceBuf tr;
#endif
};

// CAUSAL: the rows of a context-fill chunk, masked by their position instead of by ancestor bits.
template <int DH, bool CAUSAL>
__global__ void __launch_bounds__(ATTN_THREADS, 1) k_tree_attention_tc(const __grid_constant__ CUtensorMap tmQ,
                                                                       const __grid_constant__ SegTable tab,
                                                                       const AttnParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  AttnCtl* sc = (AttnCtl*)(smem + attn::smem_bytes(DH));
  const int warp = warp_index(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    attn::ctl_init(&sc->a);
    sc->abort = 0;
    mbar_fence_init();
    tma_prefetch_desc(&tmQ);
  }
  if (warp == 1) tmem_alloc(&sc->tmem_base, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_launch_dependents();                 // not before this CTA has its tensor memory
  SPECASR_TRACE_SCOPE(p.tr, SPECASR_KIND_ATTN);
  pdl_wait();
  SPECASR_TRACE_MARK();
  const uint32_t tmem = sc->tmem_base;
  volatile int* abort = &sc->abort;
  attn::snapshot(&sc->a, tab);
  __syncthreads();

  if (warp == 0) {
    if (elect_one()) {
      int pos = 0, units = 0, L = 0, kc = 0;
      const uint64_t policy = make_evict_normal();
#pragma unroll 1
      for (int u = blockIdx.x; u < tab.units; u += gridDim.x) {
        const attn::Unit un = attn::unit_of(tab, u, p.Hkv, p.nodes_per_tile);
        if (!attn::unit_live<CAUSAL>(&sc->a, tab, un, L, kc, p.nodes_per_tile) || kc <= 0) continue;
        int32_t* status = tab.seg[un.seg].ctl + CTL_STATUS;
        auto wait = [&](void* bar, uint32_t parity) -> bool { return mbar_wait(bar, parity, abort, status); };
        if (!attn::produce<DH>(&sc->a, smem, &tmQ, tab.seg[un.seg], p.page_size, p.layer, p.Hkv, un, kc, p.group,
                               p.nodes_per_tile * p.group, pos, units, policy, wait))
          break;
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      int pos = 0, g = 0, units = 0, L = 0, kc = 0;
#pragma unroll 1
      for (int u = blockIdx.x; u < tab.units; u += gridDim.x) {
        const attn::Unit un = attn::unit_of(tab, u, p.Hkv, p.nodes_per_tile);
        if (!attn::unit_live<CAUSAL>(&sc->a, tab, un, L, kc, p.nodes_per_tile) || kc <= 0) continue;
        int32_t* status = tab.seg[un.seg].ctl + CTL_STATUS;
        auto wait = [&](void* bar, uint32_t parity) -> bool { return mbar_wait(bar, parity, abort, status); };
        if (!attn::multiply<DH>(&sc->a, smem, tmem, kc, pos, g, units, wait)) break;
      }
      attn::drain(&sc->a, pos, g, units, [&](void* bar, uint32_t parity) -> bool {
        return mbar_wait(bar, parity, abort, tab.seg[0].ctl + CTL_STATUS);
      });
    }
  } else {
    const int quad = warp & 3, half = (warp - 2) >> 2, row = quad * 32 + lane;
    int pos = 0, g = 0, L = 0, kc = 0;
#pragma unroll 1
    for (int u = blockIdx.x; u < tab.units; u += gridDim.x) {
      const attn::Unit un = attn::unit_of(tab, u, p.Hkv, p.nodes_per_tile);
      if (!attn::unit_live<CAUSAL>(&sc->a, tab, un, L, kc, p.nodes_per_tile)) continue;
      const SegDev& sg = tab.seg[un.seg];
      const int node = un.node0 + row / p.group;
      attn::RowState rs;
      rs.valid = row < p.nodes_per_tile * p.group && node < sg.n;
      const size_t out = (size_t)un.split * p.rows_alloc + (size_t)(sg.row0 + node) * p.Hq + un.kvh * p.group + row % p.group;
      if (kc <= 0) {
        if (rs.valid && half == 0) p.attML[out] = make_float2(-INFINITY, 0.f);
        continue;
      }
      rs.node = node;
      if constexpr (!CAUSAL) {
#pragma unroll
        for (int w = 0; w < 4; ++w) rs.anc[w] = rs.valid ? p.anc[(size_t)(sg.row0 + node) * 4 + w] : 0ull;
      }
      int32_t* status = sg.ctl + CTL_STATUS;
      auto wwait = [&](void* bar, uint32_t parity) -> bool {   // one verdict per warp: TMEM accesses are warp-wide
        return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, abort, status) ? 1 : 0) != 0;
      };
      attn::soften<DH, CAUSAL>(&sc->a, smem, tmem, kc, un.k_begin, L, p.scale_log2, rs, quad, half, pos, g, p.attO + out * DH,
                       p.attML + out, wwait);
    }
  }

  __syncwarp();                            // one lane of warps 0 and 1 had a role: what follows is meant for whole warps
  tc_fence_before();
  __syncthreads();
  if (*abort) {
    // give copies still in flight time to land before the shared memory is handed back
    for (int i = 0; i < 64; ++i) __nanosleep(20000);
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

constexpr size_t smem_total(int dh) { return attn::smem_bytes(dh) + sizeof(AttnCtl) + 1024; }

template <int DH, bool CAUSAL>
void launch_dh(specasr_kv* wk, const SegTable& t, int layer, cudaStream_t s) {
  const specasr_model* m = wk->m;
  const specasr_model_config& c = m->cfg;
  AttnParams p;
  memset(&p, 0, sizeof(p));
  p.anc = wk->ws.anc;
  const Workspace& ws = CAUSAL ? wk->fill : wk->ws;
  p.attO = ws.attO;
  p.attML = ws.attML;
  p.rows_alloc = (size_t)ws.rows * c.n_heads;
  p.page_size = c.page_size;
  p.layer = layer;
  p.Hq = c.n_heads;
  p.Hkv = c.n_kv_heads;
  p.group = c.n_heads / c.n_kv_heads;
  p.nodes_per_tile = 128 / p.group;
  p.scale_log2 = 1.4426950408889634f / sqrtf((float)DH);
#ifdef SPECASR_TRACE
  p.tr = wk->trace;
#endif
  LaunchScope scope(wk, SPECASR_KIND_ATTN, s);
  launch_pdl(k_tree_attention_tc<DH, CAUSAL>, dim3(t.units < m->n_sm ? t.units : m->n_sm), dim3(ATTN_THREADS), smem_total(DH), s,
             CAUSAL ? wk->fill_Q : wk->tm_Q, t, p);
}

}  // namespace

cudaError_t attention_tc_setup() {
  cudaError_t e = cudaSuccess;
  auto raise = [&](auto kernel, int dh) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_total(dh));
  };
  raise(k_tree_attention_tc<64, false>, 64);
  raise(k_tree_attention_tc<64, true>, 64);
  raise(k_tree_attention_tc<128, false>, 128);
  raise(k_tree_attention_tc<128, true>, 128);
  return e;
}

bool attention_tc_supported(const specasr_model* m) {
  const specasr_model_config& c = m->cfg;
  const int group = c.n_heads / c.n_kv_heads;
  return c.gemm_path == 0 && (c.head_dim == 64 || c.head_dim == 128) && c.page_size % 16 == 0 && group <= 128;
}

// Time of the busiest CTA over a context-fill chunk cut into ranges of `per` positions, by the order in which units are dealt
// out: the later a row tile, the more positions it sees.  (Some thirty sizes are tried per chunk, on the host, while the GPU has
// two small kernels to run: 18 us on 1B, 13 on 13B; unit by unit 51 and 63.)
template <typename Cost>
static float causal_load(const specasr_model* m, const SegTable& tab, int len, int nodes_per_tile, int per, Cost&& cost) {
  constexpr int MAX_SM = 256;
  const int n = tab.seg[0].n, row_tiles = (n + nodes_per_tile - 1) / nodes_per_tile, heads = m->cfg.n_kv_heads;
  const int sms = m->n_sm < MAX_SM ? m->n_sm : MAX_SM;
  const float full = cost(per);
  float load[MAX_SM] = {}, busiest = 0.f;
  int cta = 0;
  for (int k0 = 0; k0 < len + n; k0 += per)
    for (int t = 0; t < row_tiles; ++t) {
      const int rows = n < (t + 1) * nodes_per_tile ? n : (t + 1) * nodes_per_tile, keys = len + rows - k0;
      const float us = keys >= per ? full : keys > 0 ? cost(keys) : 0.f;      // the same for every head
      for (int left = heads; left > 0;) {
        const int run = left < sms - cta ? left : sms - cta;
        for (int i = cta; i < cta + run; ++i) load[i] += us;
        left -= run;
        cta = cta + run == sms ? 0 : cta + run;
      }
    }
  for (int i = 0; i < sms; ++i) busiest = load[i] > busiest ? load[i] : busiest;
  return busiest;
}

// Cuts every utterance's cache (tab->seg[b].n rows on top of up to len_upper[b] positions) into units of one common
// size.  The size is the cheapest by a linear model of a CTA's time: what a unit costs whatever its length (first loads,
// first scores, output), what a chunk of 64 keys costs, and what every further partial output of a row costs the merge.
void attention_tc_plan(const specasr_model* m, SegTable* tab, const int* len_upper, int max_splits) {
  const specasr_model_config& c = m->cfg;
  const int nodes_per_tile = 128 / (c.n_heads / c.n_kv_heads);
  const float per_chunk = c.head_dim == 128 ? 1.05f : 0.7f, per_unit = 3.0f, per_split = 0.2f;     // us
  int longest = 16, tiles[SPECASR_MAX_BATCH], len[SPECASR_MAX_BATCH];
  for (int b = 0; b < tab->count; ++b) {
    len[b] = len_upper[b] + tab->seg[b].n;
    tiles[b] = c.n_kv_heads * ((tab->seg[b].n + nodes_per_tile - 1) / nodes_per_tile);
    if (len[b] > longest) longest = len[b];
  }
  longest = (longest + 15) & ~15;
  int best = longest;
  float best_cost = 1e30f;
  int per = ((longest + max_splits - 1) / max_splits + 15) & ~15;
  for (bool more = true; more;) {
    if (per >= longest) {
      per = longest;
      more = false;
    }
    int units = 0;
    for (int b = 0; b < tab->count; ++b) units += tiles[b] * ((len[b] + per - 1) / per);
    const int rounds = (units + m->n_sm - 1) / m->n_sm;
    // a short last chunk costs less than a full one, but not in proportion
    auto chunks = [](int keys) { return 0.7f * keys / 64.f + 0.3f * ((keys + 63) / 64); };
    const float busiest = tab->causal ? causal_load(m, *tab, len_upper[0], nodes_per_tile, per, [&](int keys) { return per_unit + per_chunk * chunks(keys); })
                                      : rounds * (per_unit + per_chunk * chunks(per));
    const float cost = busiest + per_split * ((longest + per - 1) / per);
    if (cost < best_cost) {
      best_cost = cost;
      best = per;
    }
    per += per < 512 ? 16 : 64;
  }
  tab->splits = 1;
  tab->units = 0;
  for (int b = 0; b < tab->count; ++b) {
    SegDev& sg = tab->seg[b];
    sg.chunk = best;
    sg.splits = (len[b] + best - 1) / best;
    sg.unit0 = tab->units;
    tab->units += tiles[b] * sg.splits;
    if (sg.splits > tab->splits) tab->splits = sg.splits;
  }
}

// Tensor maps of the rotated queries and of the two pools, as the kernel above walks them.
bool attention_tc_make_maps(specasr_kv* kv) {
  const specasr_model* m = kv->m;
  const specasr_model_config& c = m->cfg;
  const int group = c.n_heads / c.n_kv_heads;
  const uint64_t dh = c.head_dim;
  {  // Q: [plane][node][head][dh]; box = 64 of dh, the `group` heads of one KV head, 128 / group nodes
    uint64_t dims[4] = {dh, (uint64_t)c.n_heads, (uint64_t)kv->n_alloc, 2};
    uint64_t strides[3] = {dh * 2, (uint64_t)m->q_dim * 2, (uint64_t)kv->n_alloc * m->q_dim * 2};
    uint32_t box[4] = {64, (uint32_t)group, (uint32_t)(128 / group), 1};
    if (!make_tensor_map_nd(&kv->tm_Q, kv->ws.Q, 4, dims, strides, box)) return false;
    dims[2] = (uint64_t)kv->fill.rows;
    strides[2] = (uint64_t)kv->fill.rows * m->q_dim * 2;
    if (kv->fill.rows > 0 && !make_tensor_map_nd(&kv->fill_Q, kv->fill.Q, 4, dims, strides, box)) return false;
  }
  const uint64_t ps = c.page_size;
  // pools: [layer and page and kv head][plane][slot][dh]; box = 64 of dh, 16 slots (any page size is a multiple), both planes
  uint64_t dims[4] = {dh, ps, 2, (uint64_t)c.n_layers * kv->n_pages * c.n_kv_heads};
  uint64_t strides[3] = {dh * 2, ps * dh * 2, 2 * ps * dh * 2};
  uint32_t box[4] = {64, 16, 2, 1};
  if (!make_tensor_map_nd(&kv->tm_K, kv->k_pool, 4, dims, strides, box) ||
      !make_tensor_map_nd(&kv->tm_V, kv->v_pool, 4, dims, strides, box))
    return false;
  // the kernel reads the pool descriptors through the utterance table, i.e. from global memory
  cudaError_t e = cudaMemcpy(kv->ws.tmKV, &kv->tm_K, sizeof(CUtensorMap), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(kv->ws.tmKV + 1, &kv->tm_V, sizeof(CUtensorMap), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    set_error("attention descriptors: %s", cudaGetErrorString(e));
    return false;
  }
  return true;
}

void launch_tree_attention_tc(specasr_kv* wk, const SegTable& t, int layer, cudaStream_t s) {
  if (t.causal) {
    if (wk->m->cfg.head_dim == 64) launch_dh<64, true>(wk, t, layer, s);
    else launch_dh<128, true>(wk, t, layer, s);
  } else {
    if (wk->m->cfg.head_dim == 64) launch_dh<64, false>(wk, t, layer, s);
    else launch_dh<128, false>(wk, t, layer, s);
  }
}
