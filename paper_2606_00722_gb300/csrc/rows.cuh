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
  // The inner loops load without predicates: lanes beyond the row read its last
  // words instead, and their masks are zero (valid()).
  __device__ static __forceinline__ int word(int q, int W) {  // first word of this lane's piece q
    return min(li() * KW + q, W - 4);
  }
  __device__ static __forceinline__ void load_any(const uint32_t* p, int W, uint32_t (&v)[KW]) {
#pragma unroll
    for (int q = 0; q < KW; q += 4) {
      const uint4 x = *reinterpret_cast<const uint4*>(p + word(q, W));
      v[q] = x.x;
      v[q + 1] = x.y;
      v[q + 2] = x.z;
      v[q + 3] = x.w;
    }
  }
  __device__ static __forceinline__ void load_shared_any(uint32_t addr, int W, uint32_t (&v)[KW]) {
#pragma unroll
    for (int q = 0; q < KW; q += 4) {
      const uint4 x = gs_lds4(addr + (uint32_t)word(q, W) * 4u);
      v[q] = x.x;
      v[q + 1] = x.y;
      v[q + 2] = x.z;
      v[q + 3] = x.w;
    }
  }
  __device__ static __forceinline__ void valid(uint32_t (&v)[KW], int W) {
#pragma unroll
    for (int q = 0; q < KW; q += 4)
      if (li() * KW + q >= W) v[q] = v[q + 1] = v[q + 2] = v[q + 3] = 0u;
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
  // w): ORs the set's EXP_NT rows, shared out among the lane groups, several in
  // flight each.  Wide rows are too large to keep EXP_NT in shared memory, and
  // a row from L2 costs about as much as testing 30 items: sets of more than
  // kRowSetMax test every item's next symbol instead (next_t, lanes on
  // consecutive words; scr: one row of shared scratch).  random-stress-1024
  // grammar, 4 x 96: forward charts 55 -> 44 ms, good masks 22 -> 18 ms.  The
  // warp walks keep or_rows: many of them share the rows in L1, and the item
  // test took their checks from 37 to 50 ms.
  static constexpr int kRowSetMax = 12;
  __device__ static __forceinline__ void waiting_on(uint32_t set, const uint32_t* exp_nt, const int16_t* next_t,
                                                    uint32_t* scr, int W, int VW, uint32_t (&v)[KW]) {
    if constexpr (KW == 8) {
      if (__reduce_add_sync(0xffffffffu, (unsigned)__popc(set)) > kRowSetMax) {
        const int lane = threadIdx.x & 31;
        if (lane < VW) scr[lane] = set;
        __syncwarp();
        uint32_t acc[KW];
#pragma unroll
        for (int i = 0; i < KW; ++i) acc[i] = 0u;
        for (int b = 0; b < 32; ++b) {
#pragma unroll
          for (int i = 0; i < KW; ++i) {
            const int w = lane + 32 * i;
            const int s = w < W ? next_t[b * W + w] : -1;
            if (s >= 0) acc[i] |= ((scr[s >> 5] >> (s & 31)) & 1u) << b;
          }
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < KW; ++i)
          if (lane + 32 * i < W) scr[lane + 32 * i] = acc[i];
        __syncwarp();
        load(scr, W, v);
        __syncwarp();
        return;
      }
    }
    or_rows(set, exp_nt, W, VW, v);
  }
  // v = the OR of the set's rows of table P ([V][W])
  __device__ static __forceinline__ void or_rows(uint32_t set, const uint32_t* P, int W, int VW, uint32_t (&v)[KW]) {
    constexpr int F = KW == 4 ? 4 : 2;
    uint32_t share = 0;
#pragma unroll
    for (int b = 0; b < 32; b += S::NG) share |= 1u << b;
    share <<= gi();
#pragma unroll
    for (int i = 0; i < KW; ++i) v[i] = 0u;
    for (int w = 0; w < VW; ++w) {
      uint32_t m = __shfl_sync(0xffffffffu, set, w) & share;
      while (m) {
        uint32_t x[F][KW];
        int b = 0;
#pragma unroll
        for (int u = 0; u < F; ++u) {  // the last one again when there are fewer
          b = m ? __ffs(m) - 1 : b;
          m &= m - 1;
          load_any(P + (size_t)((w << 5) + b) * W, W, x[u]);
        }
#pragma unroll
        for (int u = 0; u < F; ++u)
#pragma unroll
          for (int i = 0; i < KW; ++i) v[i] |= x[u][i];
      }
      __syncwarp();
    }
    valid(v, W);
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

// The same for the complete items, the first four pairs of a nonterminal's
// list in one place: no loop unless its items lie in more than four words.
__device__ __forceinline__ uint32_t warp_completed(const uint32_t* row, const uint2* w4, const uint4* m4,
                                                   const int32_t* off, const uint2* lst, int V, int VW) {
  const int lane = threadIdx.x & 31;
  uint32_t mine = 0;
  for (int v = 0; v < VW; ++v) {
    const int A = (v << 5) + lane;
    bool hit = false;
    if (A < V) {
      const uint2 w = w4[A];
      const uint4 m = m4[A];
      hit = ((row[w.x & 255u] & m.x) | (row[(w.x >> 8) & 255u] & m.y) | (row[(w.x >> 16) & 255u] & m.z) |
             (row[w.x >> 24] & m.w)) != 0;
      if (w.y && !hit)
        for (int q = off[A] + 4, e = off[A + 1]; q < e && !hit; ++q) hit = (row[lst[q].x] & lst[q].y) != 0;
    }
    const uint32_t b = __ballot_sync(0xffffffffu, hit);
    if (lane == v) mine = b;
  }
  return mine;
}

// Warp: every nonterminal whose completion follows from one of the set (lane
// v < VW holds word v), by the rows of `follow` ([V][VW], transitively
// closed: a nonterminal already reached adds nothing).
__device__ __forceinline__ uint32_t warp_follow(uint32_t set, const uint32_t* follow, int VW) {
  const int lane = threadIdx.x & 31;
  uint32_t acc = 0;
  for (int v = 0; v < VW; ++v) {
    uint32_t m = __shfl_sync(0xffffffffu, set, v);
    for (;;) {
      m &= ~__shfl_sync(0xffffffffu, acc, v);
      if (!m) break;
      const int A = (v << 5) + __ffs(m) - 1;
      m &= m - 1;
      if (lane < VW) acc |= follow[(size_t)A * VW + lane];
    }
  }
  return acc;
}

}  // namespace epic
