// Item bitset rows in a warp's registers: the layout and the operations that
// every walk and the good pass share.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace epic {

// How a row of W words (a multiple of 4) lies in a warp: LR lanes hold KW
// consecutive words each; the warp's 32 / LR lane groups work on different
// entries, or hold copies of one row.
template <int LRv, int KWv>
struct RowShape {
  static constexpr int LR = LRv, KW = KWv, NG = 32 / LRv;
};
using RowNarrow = RowShape<4, 4>;   // W <= 16
using RowMid = RowShape<16, 4>;     // W <= 64
using RowWide = RowShape<32, 8>;    // W <= 256
// call f with the shape of rows of W words
template <class F>
inline void with_row_shape(int W, F f) {
  if (W <= 16)
    f(RowNarrow{});
  else if (W <= 64)
    f(RowMid{});
  else
    f(RowWide{});
}

__device__ __forceinline__ uint32_t gs_saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16 bytes of a shared row that other warps may be writing
__device__ __forceinline__ uint4 gs_lds4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr));
  return v;
}
__device__ __forceinline__ void gs_red_or(uint32_t addr, uint32_t v) {
  asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// A row's words of this lane: KW words from word li * KW of p (words beyond W
// read as zero), the shift to the next item (item (p, d) -> (p, d + 1)), and
// the shift back.
template <class S>
struct RowRegs {
  static constexpr int KW = S::KW, LR = S::LR;
  __device__ static __forceinline__ int li() { return (threadIdx.x & 31) & (LR - 1); }
  __device__ static __forceinline__ int gi() { return (threadIdx.x & 31) / LR; }
  __device__ static __forceinline__ void load(const uint32_t* p, int W, uint32_t (&v)[KW]) {
    const int w0 = li() * KW;
#pragma unroll
    for (int q = 0; q < KW; q += 4) {
      uint4 x = make_uint4(0u, 0u, 0u, 0u);
      if (w0 + q < W) x = *reinterpret_cast<const uint4*>(p + w0 + q);
      v[q] = x.x;
      v[q + 1] = x.y;
      v[q + 2] = x.z;
      v[q + 3] = x.w;
    }
  }
  __device__ static __forceinline__ void load_shared(uint32_t addr, int W, uint32_t (&v)[KW]) {
    const int w0 = li() * KW;
#pragma unroll
    for (int q = 0; q < KW; q += 4) {
      uint4 x = make_uint4(0u, 0u, 0u, 0u);
      if (w0 + q < W) x = gs_lds4(addr + (uint32_t)(w0 + q) * 4u);
      v[q] = x.x;
      v[q + 1] = x.y;
      v[q + 2] = x.z;
      v[q + 3] = x.w;
    }
  }
  __device__ static __forceinline__ void store(uint32_t* p, int W, const uint32_t (&v)[KW]) {
    const int w0 = li() * KW;
#pragma unroll
    for (int q = 0; q < KW; q += 4)
      if (w0 + q < W) *reinterpret_cast<uint4*>(p + w0 + q) = make_uint4(v[q], v[q + 1], v[q + 2], v[q + 3]);
  }
  __device__ static __forceinline__ void shift_up(uint32_t (&v)[KW], int k = 1) {  // by k < 32 items
    uint32_t prev = __shfl_up_sync(0xffffffffu, v[KW - 1], 1, LR);
    if (li() == 0) prev = 0u;
#pragma unroll
    for (int i = KW - 1; i > 0; --i) v[i] = __funnelshift_l(v[i - 1], v[i], k);
    v[0] = __funnelshift_l(prev, v[0], k);
  }
  __device__ static __forceinline__ void shift_down(const uint32_t (&r)[KW], uint32_t (&s)[KW]) {
    uint32_t next = __shfl_down_sync(0xffffffffu, r[0], 1, LR);
    if (li() == LR - 1) next = 0u;
#pragma unroll
    for (int i = 0; i + 1 < KW; ++i) s[i] = __funnelshift_r(r[i], r[i + 1], 1);
    s[KW - 1] = __funnelshift_r(r[KW - 1], next, 1);
  }
  // lane groups' partial rows into every group
  __device__ static __forceinline__ void join(uint32_t (&v)[KW]) {
#pragma unroll
    for (int off = LR; off < 32; off <<= 1)
#pragma unroll
      for (int i = 0; i < KW; ++i) v[i] |= __shfl_xor_sync(0xffffffffu, v[i], off);
  }
  // v = the items waiting on a nonterminal of the set (lane w < VW holds word
  // w): the groups share out the EXP_NT rows, two in flight each
  __device__ static __forceinline__ void waiting_on(uint32_t set, const uint32_t* exp_nt, int W, int VW,
                                                    uint32_t (&v)[KW]) {
    uint32_t share = 0;
#pragma unroll
    for (int b = 0; b < 32; b += S::NG) share |= 1u << b;
    share <<= gi();
#pragma unroll
    for (int i = 0; i < KW; ++i) v[i] = 0u;
    for (int w = 0; w < VW; ++w) {
      uint32_t m = __shfl_sync(0xffffffffu, set, w) & share;
      while (m) {
        const int b0 = __ffs(m) - 1;
        m &= m - 1;
        const int b1 = m ? __ffs(m) - 1 : b0;
        m &= m - 1;
        uint32_t x[KW], y[KW];
        load(exp_nt + (size_t)((w << 5) + b0) * W, W, x);
        load(exp_nt + (size_t)((w << 5) + b1) * W, W, y);
#pragma unroll
        for (int i = 0; i < KW; ++i) v[i] |= x[i] | y[i];
      }
      __syncwarp();
    }
    join(v);
  }
  // Closure of r under item i -> i + 1 for i in the advance mask (mode 0:
  // nullable_next, 1: next_any), by doubling: step s adds i + 2^s for every i
  // in r that starts a run of 2^s advanceable items (adv_pow); steps in
  // increasing order reach every i + d with d < 2^steps, which covers the
  // longest production.
  __device__ static __forceinline__ void advance(uint32_t (&r)[KW], const uint32_t* adv_pow, int mode, int steps,
                                                 int any_nullable, int W) {
    if (mode == 0 && !any_nullable) return;  // nothing is skipped
    for (int st = 0; st < steps; ++st) {
      uint32_t v[KW];
      load(adv_pow + ((size_t)mode * steps + st) * W, W, v);
#pragma unroll
      for (int i = 0; i < KW; ++i) v[i] &= r[i];
      const int k = 1 << st;
      if (k < 32) {
        shift_up(v, k);
#pragma unroll
        for (int i = 0; i < KW; ++i) r[i] |= v[i];
      } else {  // 32 items (rhs <= 62): word w takes word w - 1
        const uint32_t prev = __shfl_up_sync(0xffffffffu, v[KW - 1], 1, LR);
#pragma unroll
        for (int i = KW - 1; i > 0; --i) r[i] |= v[i - 1];
        if (li() > 0) r[0] |= prev;
      }
    }
  }
};

// Warp: the nonterminals with an item of the (word, mask) lists in `row`
// (readable by every lane); lane v < VW returns word v of the set.
__device__ __forceinline__ uint32_t warp_ntset(const uint32_t* row, const int32_t* off, const uint2* lst, int V,
                                               int VW) {
  const int lane = threadIdx.x & 31;
  uint32_t mine = 0;
  for (int v = 0; v < VW; ++v) {
    const int A = (v << 5) + lane;
    bool hit = false;
    if (A < V)
      for (int q = off[A], e = off[A + 1]; q < e && !hit; ++q) {
        const uint2 p = lst[q];
        hit = (row[p.x] & p.y) != 0;
      }
    const uint32_t b = __ballot_sync(0xffffffffu, hit);
    if (lane == v) mine = b;
  }
  return mine;
}

}  // namespace epic
