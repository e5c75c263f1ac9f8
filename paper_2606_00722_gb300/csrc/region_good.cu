// Checks by region, step 2: the good-item masks of each forward chart, with
// the launcher.
#include <cuda_runtime.h>

#include "launch.h"
#include "region.cuh"

namespace epic {

constexpr int kGoodWarps = 16;          // per CTA
constexpr int kGoodEdges = 32;          // out-edges whose label masks are held at once
constexpr int kGoodMaxRounds = 1 << 18; // in-column rounds (each makes at least one item good)

// Dynamic shared memory of the good pass (byte offsets).
struct GoodPlan {
  uint32_t o_masks;              // next_any [W]
  uint32_t o_cpl_off, o_cpl;     // complete items by nonterminal
  uint32_t o_wait_off, o_wait;   // waiting items by nonterminal
  uint32_t o_exp;                // EXP_NT rows; 0: read from global memory
  uint32_t o_next;               // DevGrammar::next_t (wide rows); 0: read from global memory
  uint32_t o_fol;                // DevGrammar::follow; 0: read from global memory
  uint32_t o_col;                // column offsets [nmax + 1]
  uint32_t o_org;                // origins of the open column's entries (uint16)
  uint32_t o_scr;                // per-warp scratch, scr words each
  uint32_t o_cmp;                // per-warp list of a batch's active lanes
  uint32_t o_lbl;                // label masks of a chunk of out-edges
  uint32_t o_loc;                // entry of each origin in the open column (uint16), 0xFFFF none
  uint32_t o_chg, o_nxt, o_open; // bitmaps over the open column's entries
  uint32_t o_fold;               // per successor: something completes there
  uint32_t o_sux;                // items waiting on what completes at a successor; sux rows
  uint32_t o_row, o_gnt;         // good masks, and completed nonterminals not known good, of the open column; rows rows
  int sux, rows;
  // words of a warp's scratch: a row, or a nonterminal set.  Sets can be the
  // longer of the two: nonterminals keep their declared numbers, rows hold the
  // items that trimming leaves.
  int scr;
  uint32_t bytes;
};

static GoodPlan good_plan(const DevGrammar& g, int nmax) {
  auto r = [](size_t b) { return (b + 15) & ~(size_t)15; };
  const size_t limit = g.W <= 16 ? (size_t)108 * 1024 : (size_t)220 * 1024;
  GoodPlan p;
  size_t o = 0;
  auto put = [&](size_t bytes) {
    const size_t at = o;
    o += r(bytes);
    return (uint32_t)at;
  };
  p.o_masks = put((size_t)g.W * 4);
  p.o_cpl_off = put((size_t)(g.V + 1) * 4);
  p.o_cpl = put((size_t)g.n_cpl * 8);
  p.o_wait_off = put((size_t)(g.V + 1) * 4);
  p.o_wait = put((size_t)g.n_wait * 8);
  p.scr = g.W > g.VW ? g.W : (g.VW + 3) / 4 * 4;
  p.o_scr = put((size_t)kGoodWarps * p.scr * 4);
  p.o_cmp = put((size_t)kGoodWarps * 32 * 4);
  p.o_lbl = put((size_t)kGoodEdges * g.W * 4);
  p.o_loc = put((size_t)nmax * 2);
  const size_t bm = (size_t)((nmax + 31) / 32) * 4;
  p.o_chg = put(bm);
  p.o_nxt = put(bm);
  p.o_open = put(bm);
  p.o_fold = put((size_t)nmax * 4);
  p.o_col = put((size_t)(nmax + 1) * 4);
  p.o_org = put((size_t)nmax * 2);
  const size_t fol = (size_t)4 * g.V * g.VW * 4, nx = (size_t)64 * g.W;
  p.o_fol = fol <= 16 * 1024 ? put(fol) : 0;
  p.o_next = g.W > 64 ? put(nx) : 0;
  const size_t ex = (size_t)g.V * g.W * 4, per_row = (size_t)(2 * g.W + g.VW) * 4;
  p.o_exp = o + r(ex) + 64 * per_row <= limit ? put(ex) : 0;
  const size_t left = limit > o + 64 ? limit - o - 64 : 0;
  long long rows = (long long)(left / per_row);
  rows = rows > nmax ? nmax : (rows > 1024 ? 1024 : rows);
  p.sux = p.rows = (int)rows;
  p.o_sux = put((size_t)rows * g.W * 4);
  p.o_row = put((size_t)rows * g.W * 4);
  p.o_gnt = put((size_t)rows * g.VW * 4);
  p.bytes = (uint32_t)o;
  return p;
}

// ---- the CTAs of a cluster that share one sequence
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// barrier of the cluster's threads (of the CTA when it is alone)
__device__ __forceinline__ void good_sync(int C) {
  if (C == 1) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}
// the address in CTA `rank` of the shared variable at addr here
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ uint4 peer_load4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ uint32_t peer_load(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void peer_store(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void peer_or(uint32_t addr, uint32_t v) {
  asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// a row in global memory that another SM wrote in this kernel: past L1
template <class S>
__device__ __forceinline__ void load_row_l2(const uint32_t* p, int W, uint32_t (&v)[S::KW]) {
  const int w0 = RowRegs<S>::li() * S::KW;
#pragma unroll
  for (int q = 0; q < S::KW; q += 4) {
    uint4 x = make_uint4(0u, 0u, 0u, 0u);
    if (w0 + q < W) x = __ldcg(reinterpret_cast<const uint4*>(p + w0 + q));
    v[q] = x.x;
    v[q + 1] = x.y;
    v[q + 2] = x.z;
    v[q + 3] = x.w;
  }
}

// Row in registers (a copy in every lane group, or one per group):
// r |= bits & M & (r shifted down) until stable -- an item is good when it may
// advance within its own row and the advanced item is good.
template <class S>
__device__ __forceinline__ void good_in_row(uint32_t (&r)[S::KW], const uint32_t (&bits)[S::KW],
                                            const uint32_t (&M)[S::KW]) {
  bool some = false;
#pragma unroll
  for (int i = 0; i < S::KW; ++i) some |= (bits[i] & M[i] & ~r[i]) != 0;
  if (!__any_sync(0xffffffffu, some)) return;
  for (int it = 0; it < 64; ++it) {
    uint32_t s[S::KW];
    RowRegs<S>::shift_down(r, s);
    bool ch = false;
#pragma unroll
    for (int i = 0; i < S::KW; ++i) {
      const uint32_t add = bits[i] & M[i] & s[i] & ~r[i];
      ch |= add != 0;
      r[i] |= add;
    }
    if (!__any_sync(0xffffffffu, ch)) break;
  }
}

// Block, one warp per array: a[1 .. n] becomes its inclusive prefix sums
// (a[0] = 0).
__device__ inline void warp_prefix(int32_t* a, int n) {
  const int lane = threadIdx.x & 31;
  int base = 0;
  for (int i0 = 1; i0 <= n; i0 += 32) {
    const int i = i0 + lane;
    int s = i <= n ? a[i] : 0;
    for (int off = 1; off < 32; off <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, s, off);
      if (lane >= off) s += t;
    }
    if (i <= n) a[i] = base + s;
    base += __shfl_sync(0xffffffffu, s, 31);
  }
}

// Good items of a sequence's forward chart, columns from last to first.
// Item i of entry (j, o) is good when it is present and
//  - it is the accepting item at the accept node with the start origin;
//  - an out-edge j -> j2 scans a terminal it expects (or is epsilon) and the
//    advanced item of (j2, o) is good;
//  - it waits on a nonterminal that completes from origin j at column j2
//    (j2 = j: a nullable one) and the advanced item of (j2, o) is good;
//  - j is a gap and the item advanced over any symbol is good;
//  - it is complete with left side B, and some item of column o, origin o2,
//    waiting on B has its advanced item good at (j, o2).
// The first three read later columns only (final); the in-row ones (gap,
// nullable) close each row on its own.  The last one reads rows of this
// column, and runs in rounds over the entries with complete items, all warps
// at once: a round looks at the pairs (j, o), (o, o2) whose row (j, o2)
// changed in the round before, so a pair is read again only when it can add
// something, and an entry whose completed nonterminals are all good is done.
// Rounds end when no row changes; there are as many as completions nest at
// one end node.  (One entry at a time in ascending origin order, with four
// block barriers each, left the CTA at barriers for most of the pass.)
//
// A cluster of C CTAs shares a sequence when the sequences leave SMs idle: CTA r
// takes the entries r, r + C, ... of a column and keeps their rows, which the
// others read over distributed shared memory; successors are shared out the
// same way, their masks then going through L2.  All barriers are the cluster's
// and every CTA takes the same path to them.
//
// The open column's good masks, the items waiting on what completes at each
// successor column and the grammar lists sit in shared memory; rows beyond
// the slots stay in global memory.  What is left is bound by the loads of
// other columns' rows (several in flight per warp) and the barriers per round.
template <class S, int PER_SM, bool CLUSTER>
__global__ void __launch_bounds__(32 * kGoodWarps, PER_SM)
    k_good(DevGrammar g, int B, SeqPack sp, GoodPlan p, int ctas) {
  const int C = CLUSTER ? ctas : 1;  // CTAs per sequence
  extern __shared__ __align__(16) unsigned char dyn[];
  using Row = RowRegs<S>;
  constexpr int KW = S::KW, LR = S::LR, NG = S::NG;
  constexpr int U = KW == 4 ? 4 : 2;  // rows in flight per lane group
  const int li = Row::li(), gi = Row::gi();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x, nwarps = nthr >> 5;
  const int W = g.W, VW = g.VW, V = g.V;
  uint32_t* next_any = (uint32_t*)(dyn + p.o_masks);
  int32_t* c_off = (int32_t*)(dyn + p.o_cpl_off);
  uint2* c_lst = (uint2*)(dyn + p.o_cpl);
  int32_t* w_off = (int32_t*)(dyn + p.o_wait_off);
  uint2* w_lst = (uint2*)(dyn + p.o_wait);
  uint32_t* scr = (uint32_t*)(dyn + p.o_scr) + (size_t)warp * p.scr;
  uint32_t* cmp = (uint32_t*)(dyn + p.o_cmp) + warp * 32;
  const uint32_t s_row = gs_saddr(dyn + p.o_row);
  const int rank = C > 1 ? (int)cluster_rank() : 0;
  uint32_t* lbl = (uint32_t*)(dyn + p.o_lbl);
  uint16_t* loc = (uint16_t*)(dyn + p.o_loc);
  uint32_t* open = (uint32_t*)(dyn + p.o_open);
  uint32_t* sfold = (uint32_t*)(dyn + p.o_fold);
  int32_t* col = (int32_t*)(dyn + p.o_col);
  uint16_t* lorg = (uint16_t*)(dyn + p.o_org);
  const uint32_t* exp_nt = g.exp_nt;
  const uint32_t* follow = g.follow;
  const int16_t* next_t = g.next_t;
  __shared__ int s_self, s_more, s_next;
  __shared__ __align__(16) uint32_t s_xall[kWMaxW], s_xpart[kWMaxW];
  // the grammar lists
  for (int i = tid; i < W; i += nthr) next_any[i] = g.next_any[i];
  for (int i = tid; i <= V; i += nthr) {
    c_off[i] = g.cpl_off[i];
    w_off[i] = g.wait_off[i];
  }
  for (int i = tid; i < g.n_cpl; i += nthr) c_lst[i] = g.cpl[i];
  for (int i = tid; i < g.n_wait; i += nthr) w_lst[i] = g.wait[i];
  if (p.o_exp) {
    uint32_t* ex = (uint32_t*)(dyn + p.o_exp);
    for (int i = tid; i < V * W; i += nthr) ex[i] = g.exp_nt[i];
    exp_nt = ex;
  }
  if (p.o_fol) {
    uint32_t* f = (uint32_t*)(dyn + p.o_fol);
    for (int i = tid; i < 4 * V * VW; i += nthr) f[i] = g.follow[i];
    follow = f;
  }
  if (p.o_next) {
    int16_t* t = (int16_t*)(dyn + p.o_next);
    for (int i = tid; i < 32 * W; i += nthr) t[i] = g.next_t[i];
    next_t = t;
  }
  for (int i = tid; i < sp.nmax; i += nthr) loc[i] = 0xFFFFu;
  __syncthreads();
  // ---- warp helpers
  // the active lanes of a batch, in order, with a value each: cmp[t] =
  // value << 5 | lane; returns how many
  auto compact = [&](bool active, int value) -> int {
    const unsigned m = __ballot_sync(0xffffffffu, active);
    __syncwarp();
    if (active) cmp[__popc(m & ((1u << lane) - 1u))] = ((uint32_t)value << 5) | (uint32_t)lane;
    __syncwarp();
    return __popc(m);
  };
  // the nonterminals that the items of row wait on
  auto waited = [&](const uint32_t(&row)[KW]) -> uint32_t {
    if (lane < LR) Row::store(scr, W, row);
    __syncwarp();
    uint32_t mine = 0;
    for (int v = 0; v < VW; ++v) {
      const int A = (v << 5) + lane;
      bool hit = false;
      if (A < V)
        for (int q = w_off[A], e = w_off[A + 1]; q < e && !hit; ++q) hit = (scr[w_lst[q].x] & w_lst[q].y) != 0;
      const uint32_t b = __ballot_sync(0xffffffffu, hit);
      if (lane == v) mine = b;
    }
    __syncwarp();
    return mine;
  };
  // the complete items whose left side is in the set
  auto completes = [&](uint32_t set, uint32_t(&c)[KW]) {
    for (int w = lane; w < W; w += 32) scr[w] = 0;
    __syncwarp();
    for (int v = 0; v < VW; ++v) {
      const uint32_t m = __shfl_sync(0xffffffffu, set, v);
      if ((m >> lane) & 1u) {
        const int A = (v << 5) + lane;
        for (int q = c_off[A]; q < c_off[A + 1]; ++q) atomicOr(&scr[c_lst[q].x], c_lst[q].y);
      }
    }
    __syncwarp();
    Row::load(scr, W, c);
    __syncwarp();
  };
  for (long long b = blockIdx.x / C; b < B; b += gridDim.x / C) {
    PH_BEGIN(t_setup);
    SeqArena a = sp.carve(b);
    int32_t* meta = a.rec.meta;
    if (meta[M_STATUS] != 1) continue;
    const int N = meta[M_NCOLS], NE = meta[M_NEDGES];
    __syncthreads();  // the sequence before is done with the offsets
    for (int j = tid; j <= N; j += nthr) col[j] = a.ws.col_off[j];
    __syncthreads();
    const int32_t* org = a.ws.org;
    const uint32_t* bits_g = a.ws.bits;
    const int start = meta[M_START], accept = meta[M_ACCEPT];
    if (rank == 0) {  // the indexes, by the first CTA
      int32_t* cur_o = a.cursor;          // [N + 1]
      int32_t* cur_s = a.cursor + N + 1;  // [N + 1]
      // edges by source and entries by origin (CSR), entry index by (column, origin)
      for (int j = tid; j <= N; j += nthr) {
        a.in_off[j] = 0;
        a.out_off[j] = 0;
        a.succ_off[j] = 0;
      }
      for (int u = tid; u < N; u += nthr) a.last_col[u] = -1;
      const size_t ntri = (size_t)N * (N + 1) / 2;
      for (size_t q = tid; q < ntri; q += nthr) a.eidx[q] = -1;
      __syncthreads();
      for (int e = tid; e < NE; e += nthr) {
        atomicAdd(&a.in_off[a.rec.e_dst[e] + 1], 1);
        atomicAdd(&a.out_off[a.rec.e_src[e] + 1], 1);
      }
      for (int j = warp; j < N; j += nwarps)
        for (long long k = col[j] + lane; k < col[j + 1]; k += 32) {
          const int o = org[k];
          a.eidx[tri_index(j, o)] = (int32_t)k;
          a.gnz[k] = 0;
          atomicAdd(&a.succ_off[o + 1], 1);
          atomicMax(&a.last_col[o], j);
        }
      __syncthreads();
      if (warp < 3) warp_prefix(warp == 0 ? a.in_off : (warp == 1 ? a.out_off : a.succ_off), N);
      __syncthreads();
      for (int j = tid; j < N; j += nthr) {
        cur_o[j] = a.out_off[j];
        cur_s[j] = a.succ_off[j];
      }
      __syncthreads();
      for (int e = tid; e < NE; e += nthr) a.out_idx[atomicAdd(&cur_o[a.rec.e_src[e]], 1)] = e;
      for (int j = warp; j < N; j += nwarps)
        for (long long k = col[j] + lane; k < col[j + 1]; k += 32) a.succ_idx[atomicAdd(&cur_s[org[k]], 1)] = j;
      __syncthreads();
    }
    good_sync(C);
    PH_END(0, t_setup);
    uint32_t* G = a.good;
    for (int j = N - 1; j >= 0; --j) {
      const int s0 = a.succ_off[j], s1 = a.succ_off[j + 1];
      const bool gap = a.rec.col_gap[j] != 0;
      const int k0 = col[j], ne = col[j + 1] - k0;
      if (ne == 0) continue;
      uint32_t* chg = (uint32_t*)(dyn + p.o_chg);
      uint32_t* nxt = (uint32_t*)(dyn + p.o_nxt);
      auto row_of = [&](int e) -> uint32_t* {
        const int slot = e / C;  // rows of this CTA's entries (e % C == rank)
        return slot < p.rows ? (uint32_t*)(dyn + p.o_row) + (size_t)slot * W : G + (size_t)(k0 + e) * W;
      };
      auto gnt_of = [&](int e) -> uint32_t* {  // overflow: the forward walk's completion record is free
        const int slot = e / C;
        return slot < p.rows ? (uint32_t*)(dyn + p.o_gnt) + (size_t)slot * VW : a.bdone + (size_t)e * VW;
      };
      auto sux_of = [&](int s) -> uint32_t* {
        return C == 1 && s < p.sux ? (uint32_t*)(dyn + p.o_sux) + (size_t)s * W : a.expn + (size_t)s * W;
      };
      auto load_sux = [&](int s, uint32_t(&v)[KW]) {
        if (C == 1)
          Row::load(sux_of(s), W, v);
        else
          load_row_l2<S>(sux_of(s), W, v);
      };
      auto load_later = [&](size_t k, uint32_t(&v)[KW]) {  // good mask of a later column's entry
        if (C == 1)
          Row::load(G + k * W, W, v);
        else
          load_row_l2<S>(G + k * W, W, v);
      };
      auto is_good = [&](int k) -> bool { return (C == 1 ? a.gnz[k] : __ldcg(a.gnz + k)) != 0; };
      // a row that its owner may be writing (bits only get set)
      auto load_good = [&](int e, uint32_t(&v)[KW]) {
        const int slot = e / C;
        if (slot < p.rows) {
          const uint32_t at = s_row + (uint32_t)slot * (uint32_t)(W * 4);
          if (C == 1) {
            Row::load_shared(at, W, v);
          } else {
            const uint32_t far = peer_addr(at, (uint32_t)(e - slot * C)) + (uint32_t)(li * KW) * 4u;
#pragma unroll
            for (int q = 0; q < KW; q += 4) {
              uint4 x = make_uint4(0u, 0u, 0u, 0u);
              if (li * KW + q < W) x = peer_load4(far + 4u * q);
              v[q] = x.x;
              v[q + 1] = x.y;
              v[q + 2] = x.z;
              v[q + 3] = x.w;
            }
          }
        } else {
#pragma unroll
          for (int i = 0; i < KW; ++i)
            v[i] = li * KW + i < W ? *(volatile const uint32_t*)(G + (size_t)(k0 + e) * W + li * KW + i) : 0u;
        }
      };
      // in-row rules of this column: the gap self-loop and nullable completions
      auto in_row = [&](uint32_t(&m)[KW], bool gp, int self_si) {
        if (gp) {
          Row::load(next_any, W, m);
        } else {
#pragma unroll
          for (int i = 0; i < KW; ++i) m[i] = 0u;
        }
        if (self_si >= 0 && sfold[self_si]) {
          uint32_t x[KW];
          load_sux(self_si, x);
#pragma unroll
          for (int i = 0; i < KW; ++i) m[i] |= x[i];
        }
      };
      // what completes from origin j at each column j2 (j2 = j included): the
      // items waiting on it, and their union over the successors after j
      PH_BEGIN(t_succ);
      if (tid == 0) {
        s_self = -1;
        s_next = 0;
      }
      for (int w = tid; w < W; w += nthr) s_xpart[w] = 0;
      for (int e = tid; e < ne; e += nthr) {
        const int o = org[k0 + e];
        loc[o] = (uint16_t)e;
        lorg[e] = (uint16_t)o;
      }
      for (int w = tid; w < ((ne + 31) >> 5); w += nthr) {
        chg[w] = 0;
        nxt[w] = 0;
        open[w] = 0;
      }
      __syncthreads();
      // s_self and sfold of every CTA may be written by the others from here on
      if (C > 1) good_sync(C);
      for (int si = s0 + warp * C + rank; si < s1; si += nwarps * C) {
        const int j2 = a.succ_idx[si];
        const uint32_t* cn = a.rec.cnt + (size_t)a.eidx[tri_index(j2, j)] * VW;
        const uint32_t set = lane < VW ? cn[lane] : 0u;
        const uint32_t f = __any_sync(0xffffffffu, set != 0) ? 1u : 0u;
        if (lane < C) {
          if (C == 1) {
            sfold[si - s0] = f;
            if (j2 == j) s_self = si - s0;
          } else {
            peer_store(peer_addr(gs_saddr(sfold + (si - s0)), lane), f);
            if (j2 == j) peer_store(peer_addr(gs_saddr(&s_self), lane), (uint32_t)(si - s0));
          }
        }
        if (f) {
          uint32_t ex[KW];
          Row::waiting_on(set, exp_nt, next_t, scr, W, VW, ex);
          if (lane < LR) {
            Row::store(sux_of(si - s0), W, ex);
            if (j2 != j) {
#pragma unroll
              for (int i = 0; i < KW; ++i)
                if (ex[i] & ~*(volatile uint32_t*)&s_xpart[min(li * KW + i, kWMaxW - 1)])
                  atomicOr(&s_xpart[li * KW + i], ex[i]);
            }
          }
        }
      }
      good_sync(C);
      for (int w = tid; w < W; w += nthr) {  // the CTAs' unions
        uint32_t u = 0;
        for (int r = 0; r < C; ++r) u |= C == 1 ? s_xpart[w] : peer_load(peer_addr(gs_saddr(s_xpart + w), r));
        s_xall[w] = u;
      }
      // A. the rules that read later columns: out-edges, a chunk at a time
      const int eb0 = a.out_off[j], eb1 = a.out_off[j + 1];
      int chunk = eb0;
      do {
        const int nc = min(kGoodEdges, eb1 - chunk);
        __syncthreads();
        for (int q = warp; q < nc; q += nwarps) {  // label masks of the chunk
          const uint32_t* L = a.rec.e_lbl + (size_t)a.out_idx[chunk + q] * 8;
          uint32_t m[KW];
#pragma unroll
          for (int i = 0; i < KW; ++i) m[i] = 0u;
          int seen = 0;
          for (int lw = 0; lw < 8; ++lw) {  // the lane groups share out the terminals
            uint32_t lm = L[lw];
            while (lm) {
              const int t = (lw << 5) + __ffs(lm) - 1;
              lm &= lm - 1;
              if ((seen++ & (NG - 1)) != gi || t >= g.T) continue;
              uint32_t x[KW];
              Row::load(g.exp_term + (size_t)t * W, W, x);
#pragma unroll
              for (int i = 0; i < KW; ++i) m[i] |= x[i];
            }
          }
          __syncwarp();
          Row::join(m);
          if (lane < LR) Row::store(lbl + (size_t)q * W, W, m);
        }
        __syncthreads();
        PH_END(1, t_succ);
        PH_BEGIN(t_a);
        // this lane's edge of the chunk
        int dst = -1;
        bool eps = true;
        if (lane < nc) {
          const int e = a.out_idx[chunk + lane];
          dst = a.rec.e_dst[e];
          for (int lw = 0; lw < 8; ++lw) eps &= a.rec.e_lbl[(size_t)e * 8 + lw] == 0u;
        }
        const unsigned epsm = __ballot_sync(0xffffffffu, eps);
        const bool first = chunk == eb0, last = chunk + nc >= eb1;
        const int self_si = s_self;
        uint32_t inrow[KW];  // in-row rules of this column: the gap self-loop and nullable completions
        in_row(inrow, gap, self_si);
        for (int e = warp * C + rank; e < ne; e += nwarps * C) {
          const size_t k = (size_t)k0 + e;
          const int o = lorg[e];
          uint32_t* Gk = row_of(e);
          uint32_t acc[KW], bits[KW];
          // the lane groups take different edges and successors, and their
          // parts are joined; `bits` is in every group
          Row::load(bits_g + k * W, W, bits);
          if (first) {
#pragma unroll
            for (int i = 0; i < KW; ++i) acc[i] = 0u;
          } else {
            Row::load(Gk, W, acc);
          }
          if (j == accept && o == start) {
#pragma unroll
            for (int i = 0; i < KW; ++i)
              if (li * KW + i == (g.accept_item >> 5)) acc[i] |= 1u << (g.accept_item & 31);
          }
          int k2 = dst >= 0 ? a.eidx[tri_index(dst, o)] : -1;
          if (k2 >= 0 && !is_good(k2)) k2 = -1;
          const int na = compact(k2 >= 0, k2);
          for (int t0 = 0; t0 < na; t0 += NG * U) {
            uint32_t gv[U][KW];
            int l[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              // this group's edge: the t-th active one (past the end: the last one again)
              const uint32_t c = cmp[min(t0 + u * NG + gi, na - 1)];
              l[u] = c & 31;
              load_later(c >> 5, gv[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
              uint32_t s[KW], m[KW];
              Row::shift_down(gv[u], s);
              const bool ep = (epsm >> l[u]) & 1u;
              Row::load(lbl + (size_t)l[u] * W, W, m);
#pragma unroll
              for (int i = 0; i < KW; ++i) acc[i] |= ep ? gv[u][i] : (s[i] & m[i]);
            }
          }
          Row::join(acc);
          if (last) {
            // the most the nested rule can make good: items waiting on a
            // nonterminal that completes from j somewhere after j
            uint32_t want[KW];
#pragma unroll
            for (int i = 0; i < KW; ++i) want[i] = bits[i] & s_xall[min(li * KW + i, kWMaxW - 1)];
            auto saturated = [&]() {
              bool left = false;
#pragma unroll
              for (int i = 0; i < KW; ++i) left |= (want[i] & ~acc[i]) != 0;
              return !__any_sync(0xffffffffu, left);
            };
            for (int sb = s0; sb < s1; sb += 32) {
              if (saturated()) break;
              const int si = sb + lane;
              int k3 = -1;
              if (si < s1 && si - s0 != self_si && sfold[si - s0]) {
                const int kk = a.eidx[tri_index(a.succ_idx[si], o)];
                if (kk >= 0 && is_good(kk)) k3 = kk;
              }
              const int n3 = compact(k3 >= 0, k3);
              for (int t0 = 0; t0 < n3; t0 += NG * U) {
                uint32_t gv[U][KW], xv[U][KW];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                  const uint32_t c = cmp[min(t0 + u * NG + gi, n3 - 1)];
                  load_later(c >> 5, gv[u]);
                  load_sux(sb + (int)(c & 31) - s0, xv[u]);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                  uint32_t s[KW];
                  Row::shift_down(gv[u], s);
#pragma unroll
                  for (int i = 0; i < KW; ++i) acc[i] |= s[i] & xv[u][i];
                }
                Row::join(acc);
                if (t0 + NG * U < n3 && saturated()) break;
              }
            }
#pragma unroll
            for (int i = 0; i < KW; ++i) acc[i] &= bits[i];
            good_in_row<S>(acc, bits, inrow);
          }
          bool nz = false;
#pragma unroll
          for (int i = 0; i < KW; ++i) nz |= acc[i] != 0;
          __syncwarp();
          if (lane < LR) Row::store(Gk, W, acc);
          if (last) {
            nz = __any_sync(0xffffffffu, nz);
            const uint32_t cn = lane < VW ? a.rec.cnt[k * VW + lane] : 0u;
            const bool cpl = __any_sync(0xffffffffu, cn != 0);
            if (lane < VW) gnt_of(e)[lane] = cn;
            if (lane == 0) {
              if (nz) {
                if (C == 1)
                  atomicOr(&chg[e >> 5], 1u << (e & 31));
                else
                  for (int r = 0; r < C; ++r) peer_or(peer_addr(gs_saddr(&chg[e >> 5]), r), 1u << (e & 31));
              }
              if (cpl) atomicOr(&open[e >> 5], 1u << (e & 31));
            }
          }
        }
        PH_END(2, t_a);
        chunk += nc;
      } while (chunk < eb1);
      // B. completions within the column, in rounds (see above)
      PH_BEGIN(t_g);
      for (int round = 0;; ++round) {
        if (tid == 0) s_more = 0;
        good_sync(C);
        const int sel = s_self;
        for (;;) {
          int e = 0;
          if (lane == 0) e = atomicAdd(&s_next, 1);
          e = __shfl_sync(0xffffffffu, e, 0) * C + rank;
          if (e >= ne) break;
          if (!((open[e >> 5] >> (e & 31)) & 1u)) continue;
          const size_t k = (size_t)k0 + e;
          const int o = lorg[e];
          uint32_t* gnt = gnt_of(e);
          uint32_t nt = lane < VW ? gnt[lane] : 0u;  // completed, not known good
          uint32_t found = 0, ex[KW];
          bool have = false;
          const int cb = col[o], ce = col[o + 1];
          for (int c0 = cb; c0 < ce; c0 += 32) {
            const int kp = c0 + lane;
            int l2 = 0xFFFF;
            if (kp < ce) l2 = loc[org[kp]];
            const bool live = l2 != 0xFFFF && ((chg[l2 >> 5] >> (l2 & 31)) & 1u);
            const int na = compact(live, l2);
            if (na == 0) continue;
            if (!have) {
              Row::waiting_on(nt, exp_nt, next_t, scr, W, VW, ex);
              have = true;
            }
            uint32_t acc[KW];
#pragma unroll
            for (int i = 0; i < KW; ++i) acc[i] = 0u;
            for (int t0 = 0; t0 < na; t0 += NG * U) {
              uint32_t pv[U][KW];
              int ee[U];
#pragma unroll
              for (int u = 0; u < U; ++u) {
                const uint32_t c = cmp[min(t0 + u * NG + gi, na - 1)];
                ee[u] = (int)(c >> 5);
                Row::load(bits_g + (size_t)(c0 + (int)(c & 31)) * W, W, pv[u]);
              }
#pragma unroll
              for (int u = 0; u < U; ++u) {
                uint32_t gv[KW], s[KW];
                load_good(ee[u], gv);
                Row::shift_down(gv, s);
#pragma unroll
                for (int i = 0; i < KW; ++i) acc[i] |= pv[u][i] & s[i];
              }
            }
#pragma unroll
            for (int i = 0; i < KW; ++i) acc[i] &= ex[i];
            Row::join(acc);
            bool any = false;
#pragma unroll
            for (int i = 0; i < KW; ++i) any |= acc[i] != 0;
            if (!__any_sync(0xffffffffu, any)) continue;
            const uint32_t nw = waited(acc) & nt;
            found |= nw;
            nt &= ~nw;
            if (!__any_sync(0xffffffffu, nt != 0)) break;  // every completed nonterminal is good
          }
          if (!__any_sync(0xffffffffu, found != 0)) continue;
          // what completes here and leads to a good one through the entry of
          // column o with origin o (which maps back to this row) is good too:
          // one lane per nonterminal looks for a good one that follows from it
          {
            const uint32_t* fo = follow + (size_t)(2 * (a.rec.col_gap[o] != 0) + (gap ? 1 : 0)) * V * VW;
            uint32_t more = 0;
            if (lane < VW) scr[lane] = found;
            __syncwarp();
            for (int v = 0; v < VW; ++v) {
              const uint32_t cand = __shfl_sync(0xffffffffu, nt, v);
              bool hit = false;
              if ((cand >> lane) & 1u)
                for (int w = 0; w < VW && !hit; ++w) hit = (fo[(size_t)((v << 5) + lane) * VW + w] & scr[w]) != 0;
              const uint32_t b2 = __ballot_sync(0xffffffffu, hit);
              if (lane == v) more = b2;
            }
            __syncwarp();
            found |= more;
            nt &= ~more;
          }
          // complete items with a good left side, and the in-row closure
          uint32_t r[KW], bits[KW], inrow[KW], cm[KW];
          uint32_t* Gk = row_of(e);
          Row::load(Gk, W, r);
          Row::load(bits_g + k * W, W, bits);
          in_row(inrow, gap, sel);
          completes(found, cm);
          bool changed = false;
#pragma unroll
          for (int i = 0; i < KW; ++i) {
            const uint32_t add = bits[i] & cm[i] & ~r[i];
            changed |= add != 0;
            r[i] |= add;
          }
          changed = __any_sync(0xffffffffu, changed);
          if (changed) good_in_row<S>(r, bits, inrow);
          if (lane < VW) gnt[lane] = nt;
          if (!__any_sync(0xffffffffu, nt != 0) && lane == 0) atomicAnd(&open[e >> 5], ~(1u << (e & 31)));
          if (changed) {
            __syncwarp();
            if (lane < LR) Row::store(Gk, W, r);
            if (lane == 0) {
              if (C == 1) {
                atomicOr(&nxt[e >> 5], 1u << (e & 31));
                s_more = 1;
              } else {
                for (int r = 0; r < C; ++r) {
                  peer_or(peer_addr(gs_saddr(&nxt[e >> 5]), r), 1u << (e & 31));
                  peer_store(peer_addr(gs_saddr(&s_more), r), 1u);
                }
              }
            }
          }
        }
        good_sync(C);
        uint32_t* t = chg;
        chg = nxt;
        nxt = t;
        const bool more = s_more != 0;
        for (int w = tid; w < ((ne + 31) >> 5); w += nthr) nxt[w] = 0;
        if (tid == 0) s_next = 0;
        if (!more) break;
        if (round > kGoodMaxRounds) {  // cannot happen; the checks would walk whole
          if (tid == 0) meta[M_STATUS] = -1;
          break;
        }
        __syncthreads();
      }
      PH_END(3, t_g);
      // the column's masks to global memory
      PH_BEGIN(t_w);
      for (int e0 = warp * NG; e0 * C < ne; e0 += nwarps * NG) {
        const int e = (e0 + gi) * C + rank;
        bool nz = false;
        if (e < ne) {
          uint32_t v[KW];
          Row::load(row_of(e), W, v);
          Row::store(G + (size_t)(k0 + e) * W, W, v);
#pragma unroll
          for (int i = 0; i < KW; ++i) nz |= v[i] != 0;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, nz);
        if (e < ne && li == 0) {
          const unsigned group = LR == 32 ? 0xffffffffu : ((1u << LR) - 1u) << (gi * LR);
          a.gnz[k0 + e] = (bal & group) ? 1 : 0;
        }
      }
      for (int e = tid; e < ne; e += nthr) loc[lorg[e]] = 0xFFFFu;
      good_sync(C);  // masks written, and nobody reads this column's rows any more
      PH_END(4, t_w);
    }
    __syncthreads();
  }
  if (C > 1) good_sync(C);  // no CTA ends while another may read its shared memory
}

// The CTAs that share a sequence: as many as leave every cluster its own SMs (a
// eighth of the SMs is spared: clusters do not fill every group of SMs).
// C-like 32 x 256: 60 ms alone, 46 with two, 30 with four; 40 x 128 19 ms alone,
// 15 with two; 64 x 256 74 and 56; 400 nonterminals 4 x 96: 44 alone, 22 with
// four, 18 with eight.  Narrow rows stay alone: their columns hold little work
// between the cluster's barriers, and the text decides (JSON 16 x 256: 9.1 ms
// alone, 7.7 with eight on one batch, 4.0 and 6.8 on another).
static int good_cluster(int B, int W, int sms) {
  int C = W <= 16 ? 1 : 8;
  while (C > 1 && (long long)B * C * 8 > 7ll * sms) C >>= 1;
  return C;
}

void launch_good(int B, cudaStream_t st, const DevGrammar& g, const SeqPack& sp) {
  const GoodPlan p = good_plan(g, sp.nmax);
  const int sms = gs_sms(), C = good_cluster(B, g.W, sms);
  auto go = [&](auto* kernel) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.bytes);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(B * C));
    cfg.blockDim = dim3(32 * kGoodWarps);
    cfg.dynamicSmemBytes = p.bytes;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = C > 1 ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, g, B, sp, p, C);
  };
  with_row_shape(g.W, [&](auto s) {
    using S = decltype(s);
    if constexpr (S::LR == 4) {
      // more sequences than SMs: two CTAs per SM at 64 registers (molecules,
      // 256 x 256: 52 ms; eight warps at 128 registers 60 ms)
      if (B > sms)
        go(k_good<S, 2, false>);
      else
        go(k_good<S, 1, false>);
    } else {
      if (C > 1)
        go(k_good<S, 1, true>);
      else
        go(k_good<S, 1, false>);
    }
  });
}

// measurement builds: this translation unit's phase counters
int phase_read_good(unsigned long long* out16, int reset) {
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
