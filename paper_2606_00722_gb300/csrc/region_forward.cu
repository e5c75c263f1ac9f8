// Checks by region, step 1: the forward chart of x per sequence (one CTA
// each, recording the graph), with its launcher.
#include <cuda_runtime.h>

#include "launch.h"
#include "region.cuh"

namespace epic {

// One CTA per sequence at every row width.  (One warp per sequence served
// narrow rows before: with the chart's open rows in shared memory and the
// origins of a column shared out among 16 warps, a CTA is the faster one there
// too.)  Two CTAs share an SM when rows have at most 16 words.
template <class S>
__global__ void __launch_bounds__(32 * kGsMaxWarps, 1)
    k_forward_gs(DevGrammar g, const LexEntry* __restrict__ table, int vocab, const int32_t* __restrict__ x, int B,
                 int n, SeqPack sp, GsPlan plan, unsigned long long* stats) {
  extern __shared__ __align__(16) unsigned char dyn[];
  GsTables tb;
  gs_stage_tables(g, dyn + kWalkSmemBytes, tb);
  for (long long b = blockIdx.x; b < B; b += gridDim.x) {
    SeqArena a = sp.carve(b);
    // the walk expects a zeroed stage and completion record
    for (size_t w = threadIdx.x; w < (size_t)sp.nmax * g.W; w += blockDim.x) a.ws.stage[w] = 0;
    for (size_t w = threadIdx.x; w < (size_t)sp.nmax * g.VW; w += blockDim.x) a.bdone[w] = 0;
    for (int p = threadIdx.x; p < n; p += blockDim.x) {
      a.rec.gap_col[p] = -1;
      a.rec.pre_col[p] = -1;
      a.rec.post_col[p] = -1;
    }
    Workspace ws;
    ws.stage = a.ws.stage;
    ws.bdone = a.bdone;
    ws.col_off = nullptr;
    ws.org = a.ws.org;
    ws.bits = a.ws.bits;
    ws.cov = nullptr;
    WalkScratch sc;
    sc.g_src = a.ws.g_src;
    sc.g_end = a.ws.g_end;
    sc.g_len = a.ws.g_len;
    sc.g_tail = (uint8_t*)a.ws.g_tail;  // [kMaxQ][16] bytes
    sc.g_lbl = a.ws.g_lbl;
    sc.g_last = a.ws.g_last;
    sc.f_q = a.ws.f_q;
    sc.f_c = a.ws.f_c;
    sc.key_q = a.ws.key_q;
    sc.ent = a.ent;
    EarleyColsGS<true, S>::place_scratch(g, plan, dyn, sc);
    const BlockRec br{a.rec.col_gap, a.rec.e_dst,   a.rec.e_src,   a.rec.e_lbl,    a.rec.cnt,
                      a.rec.gap_col, a.rec.pre_col, a.rec.post_col, a.rec.edge_cap};
    WsDims d;
    d.nmax = sp.nmax;
    d.emax = sp.emax;
    EarleyColsGS<true, S> cols(g, tb, plan, dyn, ws, d);
    cols.init(dyn);
    cols.rec = &br;
    Walk<EarleyColsGS<true, S>> walk(cols, g, table, sc, vocab);
    walk.rec = &br;
    Subst none{nullptr, nullptr, 0};
    const int r = walk.run(x + b * n, n, none);
    __syncthreads();
    for (int c = threadIdx.x; c <= walk_sh().ncols; c += blockDim.x) a.ws.col_off[c] = cols.ws.col_off[c];
    if (threadIdx.x == 0) {
      int32_t* meta = a.rec.meta;
      meta[M_NCOLS] = walk_sh().ncols;
      meta[M_NEDGES] = walk_sh().nedges;
      meta[M_START] = walk_sh().start_col;
      meta[M_ACCEPT] = walk_sh().accept_col;
      meta[M_STATUS] = r == 1 ? 1 : (r == 0 ? 0 : -1);
      meta[M_NENT] = (int)walk_sh().nent;
      atomicAdd(&stats[4], (unsigned long long)walk_sh().ncols);
      atomicAdd(&stats[5], (unsigned long long)walk_sh().nent);
    }
    __syncthreads();
  }
}

template <class S>
static void launch_forward_shape(dim3 grid, cudaStream_t st, const DevGrammar& g, const LexEntry* table, int vocab,
                              const int32_t* x, int B, int n, const SeqPack& sp, unsigned long long* stats) {
  const GsPlan p = gs_plan(g, sp.nmax, gs_limit(g.W));
  cudaFuncSetAttribute(k_forward_gs<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.bytes);
  k_forward_gs<S><<<grid, gs_threads(g.W, grid.x, gs_sms()), p.bytes, st>>>(g, table, vocab, x, B, n, sp, p, stats);
}

void launch_forward_gs(dim3 grid, cudaStream_t st, const DevGrammar& g, const LexEntry* table, int vocab,
                       const int32_t* x, int B, int n, const SeqPack& sp, unsigned long long* stats) {
  with_row_shape(g.W, [&](auto s) { launch_forward_shape<decltype(s)>(grid, st, g, table, vocab, x, B, n, sp, stats); });
}

// measurement builds: this translation unit's phase counters of the walk
int phase_read_forward(unsigned long long* out16, int reset) {
#ifdef EPIC_PHASE_TIMERS
  unsigned long long h[16];
  if (cudaMemcpyFromSymbol(h, g_phase, sizeof(h)) != cudaSuccess) return -1;
  for (int i = 0; i < 16; ++i) out16[i] += h[i];
  if (reset) {
    unsigned long long z[16] = {0};
    if (cudaMemcpyToSymbol(g_phase, z, sizeof(z)) != cudaSuccess) return -1;
  }
#else
  (void)out16;
  (void)reset;
#endif
  return 0;
}

}  // namespace epic
