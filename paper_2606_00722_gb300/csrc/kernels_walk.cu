// Whole-graph walks: one warp per validity check (kernel and launcher).
#include <cuda_runtime.h>

#define EPIC_STEP __noinline__  // column steps as calls (compile time)

#include "launch.h"

using namespace epic;

// K2-K4 (warp form): one warp per validity check; warps pull checks from a
// counter.  Each check walks the lexeme graph of x (+) (pos, tok) and runs
// bit-parallel Earley recognition over it.
// zero_stage: the workspace is a shared array with earlier contents, so each
// warp clears its own stage first (walks leave it zero).
template <class S>
__global__ void __launch_bounds__(32 * kWarpsPerCta, 2) k_validate_warp(
    DevGrammar g, const LexEntry* __restrict__ table, int vocab, const int32_t* __restrict__ x, int n,
    const int32_t* __restrict__ pos, int k, const int32_t* __restrict__ cand, int K, long long total,
    uint8_t* __restrict__ valid, WPack wp, int zero_stage, unsigned long long* counter, unsigned long long* stats) {
  __shared__ WSh shm[kWarpsPerCta];
  const int warp = threadIdx.x >> 5;
  WWs ws = wp.carve((long long)blockIdx.x * (blockDim.x >> 5) + warp);
  if (zero_stage) {
    uint4* p = reinterpret_cast<uint4*>(ws.stage);
    for (int i = threadIdx.x & 31; i < wp.nmax * (g.W / 4); i += 32) p[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
  }
  WarpWalker<S, false> walk(g, table, ws, shm[warp], wp.nmax, wp.emax, vocab);
  unsigned long long n_checks = 0, n_valid = 0, n_ovf = 0, n_bad = 0, n_cols = 0, n_ent = 0;
  for (long long jb = (long long)warp * gridDim.x + blockIdx.x; jb < total; jb = next_job(counter)) {
    long long b = jb / ((long long)k * K);
    long long j = (jb / K) % k;
    int r = walk.run(x + b * n, n, pos[b * k + j], cand[jb]);
    if ((threadIdx.x & 31) == 0) valid[jb] = r == 1 ? 1 : (r == -1 ? 2 : 0);
    ++n_checks;
    n_valid += r == 1;
    n_ovf += r == -1;
    n_bad += r == -2;
    n_cols += walk.ncols;
    n_ent += walk.nent;
  }
  if ((threadIdx.x & 31) == 0 && n_checks) {
    atomicAdd(&stats[S_CHECKS], n_checks);
    atomicAdd(&stats[S_VALID], n_valid);
    atomicAdd(&stats[S_OVERFLOW], n_ovf);
    atomicAdd(&stats[S_BAD], n_bad);
    atomicAdd(&stats[S_COLUMNS], n_cols);
    atomicAdd(&stats[S_ENTRIES], n_ent);
  }
}


namespace epic {

void launch_validate_warp(dim3 grid, dim3 block, cudaStream_t st, const DevGrammar& g, const LexEntry* table, int vocab,
                          const int32_t* x, int n, const int32_t* pos, int k, const int32_t* cand, int K,
                          long long total, uint8_t* valid, const WPack& wp, int zero_stage,
                          unsigned long long* counter, unsigned long long* stats) {
  with_row_shape(g.W, [&](auto shape) {
    k_validate_warp<decltype(shape)><<<grid, block, 0, st>>>(g, table, vocab, x, n, pos, k, cand, K, total, valid, wp,
                                                             zero_stage, counter, stats);
  });
}

int phase_read_walk(unsigned long long* out16, int reset) {
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
