// Whole-graph walks, one CTA per validity check (kernel and launcher).
#include <cuda_runtime.h>

#include "launch.h"

using namespace epic;

// One CTA per check, with the columns of gscols.cuh.  A warp alone takes a
// column's origins one after another and waits for L2 at each; sixteen warps
// take them side by side over shared-memory rows.  So a walk ends several
// times sooner, at a lower rate per SM: for batches of a few checks per SM.
// cap: chart entries per check.  zero_rows: the workspace is a shared array
// with earlier contents, so each CTA clears its stage first.
template <class S>
__global__ void __launch_bounds__(32 * kGsMaxWarps, 1)
    k_validate_cta(GsPlan plan, DevGrammar g, const LexEntry* __restrict__ table, int vocab,
                   const int32_t* __restrict__ x, int n, const int32_t* __restrict__ pos, int k,
                   const int32_t* __restrict__ cand, int K, long long total, uint8_t* __restrict__ valid, WsPack wsp,
                   long long cap, int zero_rows, unsigned long long* stats) {
  extern __shared__ __align__(16) unsigned char dyn[];
  GsTables tb;
  gs_stage_tables(g, dyn + kWalkSmemBytes, tb);
  __shared__ int s_pos[1], s_tok[1];
  Workspace ws;
  WalkScratch sc;
  wsp.carve(blockIdx.x, ws, sc);
  if (zero_rows) {
    for (int i = threadIdx.x; i < wsp.dims.nmax * g.W; i += blockDim.x) ws.stage[i] = 0;
    for (int i = threadIdx.x; i < wsp.dims.nmax * g.VW; i += blockDim.x) ws.bdone[i] = 0;
    __syncthreads();
  }
  EarleyColsGS<false, S>::place_scratch(g, plan, dyn, sc);
  WsDims d = wsp.dims;
  if (cap < d.emax) d.emax = cap;
  EarleyColsGS<false, S> cols(g, tb, plan, dyn, ws, d);
  cols.init(dyn);
  Walk<EarleyColsGS<false, S>> walk(cols, g, table, sc, vocab);
  unsigned long long n_checks = 0, n_valid = 0, n_ovf = 0, n_bad = 0, n_cols = 0, n_ent = 0;
  for (long long jb = blockIdx.x; jb < total; jb += gridDim.x) {
    const long long b = jb / ((long long)k * K), j = (jb / K) % k;
    if (threadIdx.x == 0) {
      s_pos[0] = pos[b * k + j];
      s_tok[0] = cand[jb];
    }
    __syncthreads();
    const int r = walk.run(x + b * n, n, Subst{s_pos, s_tok, 1});
    if (threadIdx.x == 0) {
      valid[jb] = r == 1 ? 1 : (r == -1 ? 2 : 0);
      ++n_checks;
      n_valid += r == 1;
      n_ovf += r == -1;
      n_bad += r == -2;
      n_cols += walk_sh().ncols;
      n_ent += walk_sh().nent;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0 && n_checks) {
    atomicAdd(&stats[S_CHECKS], n_checks);
    atomicAdd(&stats[S_VALID], n_valid);
    atomicAdd(&stats[S_OVERFLOW], n_ovf);
    atomicAdd(&stats[S_BAD], n_bad);
    atomicAdd(&stats[S_COLUMNS], n_cols);
    atomicAdd(&stats[S_ENTRIES], n_ent);
  }
}

namespace epic {

void launch_validate_cta(int ctas, cudaStream_t st, const DevGrammar& g, const LexEntry* table, int vocab,
                         const int32_t* x, int n, const int32_t* pos, int k, const int32_t* cand, int K,
                         long long total, uint8_t* valid, const WsPack& wsp, long long cap, int zero_rows,
                         unsigned long long* stats) {
  const GsPlan p = gs_plan(g, wsp.dims.nmax, gs_limit(g.W));
  with_row_shape(g.W, [&](auto shape) {
    auto* kernel = k_validate_cta<decltype(shape)>;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.bytes);
    kernel<<<ctas, gs_threads(g.W, ctas, gs_sms()), p.bytes, st>>>(p, g, table, vocab, x, n, pos, k, cand, K, total,
                                                                   valid, wsp, cap, zero_rows, stats);
  });
}

}  // namespace epic
