// Warp-level Earley walk: one warp recognizes one partial output.
//
// Same graph and chart as the CTA walk (walk.cuh / skeleton.cuh), with every
// step done by one warp and no block barrier:
//  - the open column's rows lie in the warp's global stage, which its SM's L1
//    holds (sixteen warps keep 42 KB of the 256 KB as shared memory, 2.6 KB
//    each).  Staging the rows in shared memory instead cost 24 KB per warp, so
//    that seven warps ran on an SM;
//  - the closure of a column visits every origin once, from the highest down:
//    completions from origin o only advance items of origins <= o, and the one
//    entry of column o with origin o feeds row o itself (closed in registers);
//  - a row takes a group of lanes (rows.cuh): entries are scattered 32 / LR at
//    a time, with both the entries' and the destination rows' loads in flight,
//    and a store only where a row changes;
//  - the span step groups lexings by (source, end state, terminals after the
//    first) chunk by chunk, lanes matching their keys against the groups made
//    so far.
// What bounds a walk is the chain of dependent L1 / L2 accesses of its visits;
// many walks per SM hide it.
#pragma once
#include "device.cuh"
#include "rows.cuh"

namespace epic {

// the steps of a column: calls where a file asks for them
#ifndef EPIC_STEP
#define EPIC_STEP
#endif

constexpr int kWarpsPerCta = 8;
constexpr int kWCols = 4096;    // columns per walk (graph nodes)
constexpr int kWMaxW = 256;
constexpr int kWMaxQ = 1024;

// index of (column j, origin o <= j) in a lower-triangular table
__host__ __device__ __forceinline__ size_t tri_index(int j, int o) { return (size_t)j * (j + 1) / 2 + o; }

struct WWs {  // per-walk global workspace
  uint32_t* stage;   // [nmax][W] rows of the open column (zero when idle)
  int32_t* col_off;  // [nmax + 1]
  int32_t* org;      // [emax]
  uint32_t* bits;    // [emax][W]
  int32_t* f_q;      // [kWMaxQ]
  int32_t* f_c;      // [kWMaxQ]
  int32_t* g_src;    // [kWMaxQ]
  int32_t* g_end;    // [kWMaxQ]
  int32_t* g_len;    // [kWMaxQ]
  int32_t* g_last;   // [kWMaxQ]
  int32_t* key_q;    // [kWMaxQ]  representative of each end node (span step)
  uint32_t* g_tail;  // [kWMaxQ][4]  terminals 1..12 packed 4 per word
  uint32_t* g_lbl;   // [kWMaxQ][8]  first-terminal label set
};

// What a sequence's forward chart records besides the chart: the graph's edges
// in creation order of their target, gap flags, where each position's segment
// sits in the graph, and each entry's completed nonterminals.
struct SeqRec {
  uint8_t* col_gap;    // [nmax]
  int32_t* e_dst;      // [edge_cap]
  int32_t* e_src;      // [edge_cap]
  uint32_t* e_lbl;     // [edge_cap][8] terminal set of a labelled edge, all zero = epsilon
  int32_t* gap_col;    // [n] masked position -> column of its gap
  int32_t* pre_col;    // [n] fixed position -> column before its span (gap or BEGIN)
  int32_t* post_col;   // [n] fixed position -> column after its span (gap or END)
  uint32_t* cnt;       // [emax][VW] completed nonterminals of each entry
  int32_t* meta;       // [8]: ncols, nedges, start, accept, status, nent (low), -, -
  int edge_cap;
};

struct WSh {  // per-warp shared memory
  uint32_t touched[kWCols / 32];
  alignas(16) uint32_t lbl[kWMaxW];  // items that the arrivals' labels expect
  alignas(16) uint32_t scr[kWMaxW];  // one row
  int32_t list[32];
};

__device__ __forceinline__ uint32_t wl_lane() { return threadIdx.x & 31; }

// Warp: the next job after the grid's first ones (one per warp).
__device__ __forceinline__ long long next_job(unsigned long long* counter) {
  long long j = 0;
  if (wl_lane() == 0) j = (long long)atomicAdd(counter, 1ull) + (long long)gridDim.x * (blockDim.x >> 5);
  return __shfl_sync(0xffffffffu, j, 0);
}

// Warp: out[w] = items waiting on a member of the nonterminal set nts
// (VW words, readable by every lane), for the lane's words w.  A small set
// ORs its EXP_NT rows; a large one tests each item's next symbol instead
// (both give exactly the items whose next symbol is in the set).
__device__ __forceinline__ void expn_of_set(const DevGrammar& g, const uint32_t* nts, uint32_t* out) {
  const int W = g.W, VW = g.VW;
  int cnt = 0;
  for (int v = 0; v < VW; ++v) cnt += __popc(nts[v]);
  if (cnt <= 24) {
    for (int w = wl_lane(); w < W; w += 32) {
      uint32_t acc = 0;
      for (int v = 0; v < VW; ++v) {
        uint32_t m = nts[v];
        while (m) {
          const int b = __ffs(m) - 1;
          m &= m - 1;
          acc |= g.exp_nt[(size_t)((v << 5) + b) * W + w];
        }
      }
      out[w] = acc;
    }
  } else {
    for (int w = wl_lane(); w < W; w += 32) {
      uint32_t acc = 0;
      const int i0 = w << 5;
#pragma unroll 8
      for (int b = 0; b < 32; ++b) {
        const int i = i0 + b;
        const int s = i < g.D ? g.item_next[i] - g.T : -1;
        if (s >= 0 && ((nts[s >> 5] >> (s & 31)) & 1u)) acc |= 1u << b;
      }
      out[w] = acc;
    }
  }
}

#ifdef EPIC_PHASE_TIMERS
static __device__ unsigned long long g_phase[16];  // one per translation unit
#define PH_BEGIN(v) long long v = clock64()
#define PH_END(i, v)                                              \
  do {                                                            \
    if (wl_lane() == 0) atomicAdd(&g_phase[i], clock64() - (v)); \
  } while (0)
#else
#define PH_BEGIN(v)
#define PH_END(i, v)
#endif

// S: the row shape.  EXT = true adds the base chart and the suffix mode of
// checks by region (compiled out of whole-graph walks).
template <class S, bool EXT>
class WarpWalker {
 public:
  static constexpr int KW = S::KW, LR = S::LR, NG = S::NG;
  using Row = RowRegs<S>;
  const DevGrammar& g;
  const LexEntry* table;
  WWs ws;
  WSh& sh;
  int nmax;
  long long emax;
  int vocab;
  int W, VW;
  // walk state (uniform across the warp, kept in registers)
  int ncols;
  long long nent;
  int status;  // 0 ok, 1 overflow
  int nf;
  int start_col;
  // A read-only base chart (a sequence's forward chart) holds columns
  // 0 .. base_cols-1; this walk's own columns follow with ids from base_cols.
  int base_cols = 0;
  const int32_t* b_col_off = nullptr;
  const int32_t* b_org = nullptr;
  const uint32_t* b_bits = nullptr;
  bool col_labelled = false; // the open column has a labelled arrival (else only epsilon ones)
  // Checks by region: the span step about to run is the region's last and
  // the node after it is a gap resolved by the base chart's good masks.  An
  // end node all of whose lexer states reach that gap by an epsilon edge is
  // then not closed: the gap's suffix-mode test (good masks include every
  // completion an item's closure makes, and the gap advances any waiting
  // item) gives the same answer for its rows as for their closure.
  bool defer_to_gap = false;
  // the pending lexeme at lexer state q reaches a following gap by an epsilon edge
  __device__ bool eps_into_gap(int q) const {
    const int a = g.dfa_accept[q];
    return q == 0 || g.dfa_ext[q] || (a >= 0 && g.skip[a]);
  }

  __device__ WarpWalker(const DevGrammar& g_, const LexEntry* t, WWs w, WSh& s, int nm, long long em, int voc)
      : g(g_), table(t), ws(w), sh(s), nmax(nm), emax(em), vocab(voc), W(g_.W), VW(g_.VW) {
    for (int i = wl_lane(); i < kWCols / 32; i += 32) sh.touched[i] = 0;
    __syncwarp();
  }

  // ------------------------------------------------------------ chart access
  // a column's entries: origins, rows, count
  __device__ __forceinline__ int column(int c, const int32_t*& org, const uint32_t*& bits) const {
    if (EXT && c < base_cols) {
      const int b = b_col_off[c];
      org = b_org + b;
      bits = b_bits + (size_t)b * W;
      return b_col_off[c + 1] - b;
    }
    const int oc = EXT ? c - base_cols : c, b = ws.col_off[oc];
    org = ws.org + b;
    bits = ws.bits + (size_t)b * W;
    return ws.col_off[oc + 1] - b;
  }
  __device__ bool column_empty(int c) const {
    const int32_t* o;
    const uint32_t* b;
    return column(c, o, b) == 0;
  }

  // ------------------------------------------------------------ bitmaps
  // highest touched origin below `top`, or -1
  __device__ static int highest_below(const uint32_t* touched, int top) {
    if (top <= 0) return -1;
    const int t = top - 1;
    for (int wtop = t >> 5; wtop >= 0; wtop -= 32) {
      const int w = wtop - (int)wl_lane();
      uint32_t v = (w >= 0) ? touched[w] : 0u;
      if (w == (t >> 5)) v &= (t & 31) == 31 ? 0xffffffffu : ((2u << (t & 31)) - 1u);
      const unsigned any = __ballot_sync(0xffffffffu, v != 0);
      if (any) {
        const int l = __ffs(any) - 1;
        const uint32_t vv = __shfl_sync(0xffffffffu, v, l);
        return ((wtop - l) << 5) + (31 - __clz(vv));
      }
    }
    return -1;
  }
  // The touched origins below nbits in ascending order, up to 32 at a time
  // (one bitmap word): f(count, first) with their list in sh.list.
  template <class F>
  __device__ __forceinline__ void for_touched(int nbits, F f) {
    const int nw = (nbits + 31) >> 5, lane = wl_lane();
    for (int w0 = 0; w0 < nw; w0 += 32) {
      const uint32_t v = w0 + lane < nw ? sh.touched[w0 + lane] : 0u;
      unsigned any = __ballot_sync(0xffffffffu, v != 0);
      while (any) {
        const int l = __ffs(any) - 1;
        any &= any - 1;
        const uint32_t m = __shfl_sync(0xffffffffu, v, l);
        if ((m >> lane) & 1u) sh.list[__popc(m & ((1u << lane) - 1u))] = ((w0 + l) << 5) + lane;
        __syncwarp();
        f(__popc(m));
        __syncwarp();
      }
    }
  }
  __device__ __forceinline__ void touch(int o) { atomicOr(&sh.touched[o >> 5], 1u << (o & 31)); }

  // ------------------------------------------------------------ row ops
  // What a column's visits read at every step, copied to registers once per
  // column (the walker itself may lie in local memory when its steps are
  // calls).
  struct Hot {
    int W, VW, V, steps, nullable, base_cols;
    uint32_t *stage, *touched, *scr;
    const uint32_t *adv, *complete, *exp_nt, *b_bits, *bits;
    const int32_t *cpl_off, *b_off, *b_org, *off, *org;
    const uint2 *cpl, *w4;
    const uint4* m4;
    __device__ __forceinline__ int column(int c, const int32_t*& o, const uint32_t*& x) const {
      if (EXT && c < base_cols) {
        const int b = b_off[c];
        o = b_org + b;
        x = b_bits + (size_t)b * W;
        return b_off[c + 1] - b;
      }
      const int oc = EXT ? c - base_cols : c, b = off[oc];
      o = org + b;
      x = bits + (size_t)b * W;
      return off[oc + 1] - b;
    }
  };
  __device__ __forceinline__ Hot hot() const {
    Hot h;
    h.W = W;
    h.VW = VW;
    h.V = g.V;
    h.steps = g.adv_steps;
    h.nullable = g.any_nullable;
    h.base_cols = base_cols;
    h.stage = ws.stage;
    h.touched = sh.touched;
    h.scr = sh.scr;
    h.adv = g.adv_pow;
    h.complete = g.complete;
    h.exp_nt = g.exp_nt;
    h.b_bits = b_bits;
    h.bits = ws.bits;
    h.cpl_off = g.cpl_off;
    h.b_off = b_col_off;
    h.b_org = b_org;
    h.off = ws.col_off;
    h.org = ws.org;
    h.cpl = g.cpl;
    h.w4 = g.cpl4w;
    h.m4 = g.cpl4m;
    return h;
  }

  // Scatter entries of a column into the stage: row(origin) |= bits & m,
  // shifted to the next item when SHIFT.  Entries of one column have distinct
  // origins, so lane groups never share a destination row.
  template <bool SHIFT>
  __device__ static __forceinline__ void scatter(const Hot& h, const int32_t* org, const uint32_t* bits, int ne,
                                                 const uint32_t (&m)[KW]) {
    const int W = h.W;
    constexpr int U = KW == 4 ? 4 : 2;  // steps in flight
    const int lane = wl_lane(), li = Row::li(), gi = Row::gi();
    const unsigned group = LR == 32 ? 0xffffffffu : ((1u << LR) - 1u) << (gi * LR);
    for (int c0 = 0; c0 < ne; c0 += 32) {
      const int o_t = c0 + lane < ne ? org[c0 + lane] : 0;
      const int n = min(32, ne - c0);
      for (int u0 = 0; u0 < n; u0 += U * NG) {
        uint32_t v[U][KW], q[U][KW];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int t = min(u0 + u * NG + gi, n - 1);  // past the end: the last entry again
          const int o2 = __shfl_sync(0xffffffffu, o_t, t);
          Row::load_any(bits + (size_t)(c0 + t) * W, W, v[u]);
          Row::load_any(h.stage + (size_t)o2 * W, W, q[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
          for (int i = 0; i < KW; ++i) v[u][i] &= m[i];
          if (SHIFT) Row::shift_up(v[u]);
          uint32_t nw = 0;
#pragma unroll
          for (int i = 0; i < KW; ++i) {
            nw |= v[u][i] & ~q[u][i];
            q[u][i] |= v[u][i];
          }
          const unsigned bal = __ballot_sync(0xffffffffu, nw != 0);
          if (bal) {
            const int o2 = __shfl_sync(0xffffffffu, o_t, min(u0 + u * NG + gi, n - 1));
            if (bal & group) {
              Row::store(h.stage + (size_t)o2 * W, W, q[u]);
              if (li == 0) atomicOr(&h.touched[o2 >> 5], 1u << (o2 & 31));
            }
          }
        }
      }
    }
    __syncwarp();
  }

  // ------------------------------------------------------------ columns
  __device__ int open_column() {
    if (ncols >= nmax) {
      status = 1;
      return -1;
    }
    return ncols;
  }
  __device__ EPIC_STEP void arrive(int src, bool shift) {
    col_labelled |= shift;
    const Hot h = hot();
    const int32_t* org;
    const uint32_t* bits;
    const int ne = h.column(src, org, bits);
    uint32_t m[KW];
    if (shift) {
      Row::load(sh.lbl, W, m);
      scatter<true>(h, org, bits, ne, m);
    } else {
#pragma unroll
      for (int i = 0; i < KW; ++i) m[i] = 0xffffffffu;
      Row::valid(m, h.W);
      scatter<false>(h, org, bits, ne, m);
    }
  }
  __device__ void seed(int c) {
    if (wl_lane() == 0) {
      ws.stage[(size_t)c * W + (g.start_item >> 5)] |= 1u << (g.start_item & 31);
      touch(c);
    }
    __syncwarp();
  }

  // Suffix mode (a check's nodes after its region): no predictions, and rows
  // whose origin is a base-chart column are not closed here -- whether such
  // an item leads to acceptance is read from the base chart's good masks at
  // node res_node when the column is finished (found = 1); they are not kept.
  bool suffix_mode = false;
  int res_node = -1;
  const uint32_t* good = nullptr;
  int found = 0;
  int region_start = -1;  // own start column (S' item has an own origin) or -1
  int accept_node = -1;   // the base chart's accept node

  // entry of base-chart column j with origin o, or -1
  const int32_t* b_eidx = nullptr;  // [(j (j + 1) / 2) + o] for o <= j
  __device__ long long find_base(int j, int o) const { return o > j ? -1 : (long long)b_eidx[tri_index(j, o)]; }

  // Close row o (o below the open column) with its self-loop and scatter what
  // it completes over the other entries of column o.  Every lane group holds a
  // copy of the row.
  __device__ static __forceinline__ void visit(const Hot& h, int o, int mode) {
    const int W = h.W, VW = h.VW;
    const int32_t* org;
    const uint32_t* bits;
    const int ne = h.column(o, org, bits);
    uint32_t r[KW], r0[KW], e[KW], ex[KW], cs[KW];
    Row::load(h.stage + (size_t)o * W, W, r);
    const bool self = ne > 0 && org[ne - 1] == o;  // entries are stored by ascending origin
    if (self) {
      Row::load(bits + (size_t)(ne - 1) * W, W, e);
    } else {
#pragma unroll
      for (int i = 0; i < KW; ++i) e[i] = 0u;
    }
#pragma unroll
    for (int i = 0; i < KW; ++i) {
      r0[i] = r[i];
      ex[i] = cs[i] = 0u;
    }
    uint32_t known = 0;  // lane v < VW: word v of the nonterminals completed from o
    for (int round = 0; round < 64 * kWMaxW; ++round) {
      Row::advance(r, h.adv, mode, h.steps, h.nullable, W);
      uint32_t cm[KW];
      Row::load(h.complete, W, cm);
      bool fresh = false;
#pragma unroll
      for (int i = 0; i < KW; ++i) {
        cm[i] &= r[i] & ~cs[i];
        cs[i] |= cm[i];
        fresh |= cm[i] != 0;
      }
      if (!__any_sync(0xffffffffu, fresh)) break;
      if (wl_lane() < LR) Row::store(h.scr, W, cm);
      __syncwarp();
      const uint32_t nw = (LR == 4 ? warp_ntset(h.scr, h.cpl_off, h.cpl, h.V, VW)
                                   : warp_completed(h.scr, h.w4, h.m4, h.cpl_off, h.cpl, h.V, VW)) & ~known;
      __syncwarp();
      if (!__any_sync(0xffffffffu, nw != 0)) break;
      known |= nw;
      uint32_t x[KW];
      Row::or_rows(nw, h.exp_nt, W, VW, x);
      bool ch = false;
#pragma unroll
      for (int i = 0; i < KW; ++i) {
        ex[i] |= x[i];
        x[i] &= e[i];
      }
      Row::shift_up(x);
#pragma unroll
      for (int i = 0; i < KW; ++i) {
        ch |= (x[i] & ~r[i]) != 0;
        r[i] |= x[i];
      }
      if (!__any_sync(0xffffffffu, ch)) break;
    }
    bool ch = false;
#pragma unroll
    for (int i = 0; i < KW; ++i) ch |= r[i] != r0[i];
    if (__any_sync(0xffffffffu, ch)) {
      if (wl_lane() < LR) Row::store(h.stage + (size_t)o * W, W, r);
      __syncwarp();
    }
    if (__any_sync(0xffffffffu, known != 0)) scatter<true>(h, org, bits, self ? ne - 1 : ne, ex);
  }

  __device__ EPIC_STEP void close_column(int c, bool gap) {
    const int mode = gap ? 1 : 0;
    // Origins below c, each once, highest first.  A node (not a gap) reached
    // only by epsilon edges from finished columns needs none of it: each row
    // below c is a union of rows closed under completion and advance, and so
    // is the union.  In suffix mode, base-chart origins are resolved by the
    // good masks at finish.
    if (gap || col_labelled) {
      const Hot h = hot();
      const int least = EXT && suffix_mode ? base_cols : 0;
      int o = c;
      while ((o = highest_below(h.touched, o)) >= least) visit(h, o, mode);
    }
    if (EXT && suffix_mode) return;
    // predictions at c from the nonterminals waited on in any row (the
    // prediction closures are closed under further predictions)
    uint32_t uni[KW];
#pragma unroll
    for (int i = 0; i < KW; ++i) uni[i] = 0u;
    for_touched(c + 1, [&](int cnt) {
      for (int t = Row::gi(); t < cnt; t += NG) {
        uint32_t v[KW];
        Row::load(ws.stage + (size_t)sh.list[t] * W, W, v);
#pragma unroll
        for (int i = 0; i < KW; ++i) uni[i] |= v[i];
      }
    });
    Row::join(uni);
    if (wl_lane() < LR) Row::store(sh.scr, W, uni);
    __syncwarp();
    const uint32_t vs = warp_ntset(sh.scr, g.wait_off, g.wait, g.V, VW);
    __syncwarp();
    const bool any = __any_sync(0xffffffffu, vs != 0);
    const bool seeded = (sh.touched[c >> 5] >> (c & 31)) & 1u;
    if (!any && !seeded) return;
    uint32_t r[KW], p[KW];
    Row::load(ws.stage + (size_t)c * W, W, r);
    Row::or_rows(vs, gap ? g.gap_pred : g.pred, W, VW, p);
#pragma unroll
    for (int i = 0; i < KW; ++i) r[i] |= p[i];
    // a seeded row (the walk's first column) is closed by the advance rule
    if (seeded) Row::advance(r, g.adv_pow, mode, g.adv_steps, g.any_nullable, W);
    if (wl_lane() < LR) Row::store(ws.stage + (size_t)c * W, W, r);
    if (wl_lane() == 0) touch(c);
    __syncwarp();
  }

  // Move the open column's rows into the entry store (origins ascending).  A
  // touched row is never empty.
  __device__ EPIC_STEP void finish_column(int c) {
    const int oc = c - base_cols;  // own column index
    const int gi = Row::gi(), li = Row::li();
    long long E = ws.col_off[oc];
    for_touched(c + 1, [&](int cnt) {
      // rows below the base chart in suffix mode come first (origins ascend):
      // tested and dropped
      int drop = 0;
      if (EXT && suffix_mode) drop = __popc(__ballot_sync(0xffffffffu, wl_lane() < cnt && sh.list[wl_lane()] < base_cols));
      const long long E0 = E;
      const int keep = cnt - drop;
      if (E0 + keep > emax)
        status = 1;
      else
        E = E0 + keep;
      for (int t0 = 0; t0 < cnt; t0 += NG) {
        const int t = t0 + gi;
        bool hit = false;
        if (t < cnt) {
          const int o = sh.list[t];
          uint32_t* row = ws.stage + (size_t)o * W;
          uint32_t v[KW];
          Row::load(row, W, v);
          if (t < drop) {
            const long long kf = find_base(res_node, o);
            if (kf >= 0) {
              uint32_t gv[KW];
              Row::load(good + (size_t)kf * W, W, gv);
#pragma unroll
              for (int i = 0; i < KW; ++i) hit |= (v[i] & gv[i]) != 0;
            }
          } else {
            if (EXT && suffix_mode && o == region_start && res_node == accept_node) {
#pragma unroll
              for (int i = 0; i < KW; ++i)
                hit |= li * KW + i == (g.accept_item >> 5) && ((v[i] >> (g.accept_item & 31)) & 1u);
            }
            if (!status) {
              const long long k = E0 + t - drop;
              if (li == 0) ws.org[k] = o;
              Row::store(ws.bits + (size_t)k * W, W, v);
            }
          }
#pragma unroll
          for (int i = 0; i < KW; ++i) v[i] = 0u;
          Row::store(row, W, v);
        }
        if (EXT && suffix_mode && __any_sync(0xffffffffu, hit)) found = 1;
      }
    });
    for (int w = wl_lane(); w < ((c + 32) >> 5); w += 32) sh.touched[w] = 0;
    if (wl_lane() == 0) ws.col_off[oc + 1] = (int)E;
    __syncwarp();
    nent = E;
    ncols = c + 1;
    col_labelled = false;
  }

  // abandon the open column: zero its rows
  __device__ void cleanup() {
    col_labelled = false;
    for_touched(kWCols, [&](int cnt) {
      uint32_t z[KW];
#pragma unroll
      for (int i = 0; i < KW; ++i) z[i] = 0u;
      for (int t = Row::gi(); t < cnt; t += NG) Row::store(ws.stage + (size_t)sh.list[t] * W, W, z);
    });
    for (int w = wl_lane(); w < kWCols / 32; w += 32) sh.touched[w] = 0;
    __syncwarp();
  }

  __device__ bool accepts(int c, int start) {
    const int32_t* org;
    const uint32_t* bits;
    const int ne = column(c, org, bits);
    bool f = false;
    for (int k = wl_lane(); k < ne; k += 32)
      if (org[k] == start && ((bits[(size_t)k * W + (g.accept_item >> 5)] >> (g.accept_item & 31)) & 1u)) f = true;
    return __any_sync(0xffffffffu, f);
  }

  // ------------------------------------------------------------ labels
  // sh.lbl = the items that expect a terminal of the set (the lane groups
  // share out the terminals)
  __device__ EPIC_STEP void label_set(const uint32_t* lbl8) {
    uint32_t v[KW];
#pragma unroll
    for (int i = 0; i < KW; ++i) v[i] = 0u;
    int seen = 0;
    for (int lw = 0; lw < 8; ++lw) {
      uint32_t m = lbl8[lw];
      while (m) {
        const int a = (lw << 5) + __ffs(m) - 1;
        m &= m - 1;
        if ((seen++ & (NG - 1)) != Row::gi() || a >= g.T) continue;
        uint32_t x[KW];
        Row::load(g.exp_term + (size_t)a * W, W, x);
#pragma unroll
        for (int i = 0; i < KW; ++i) v[i] |= x[i];
      }
    }
    __syncwarp();
    Row::join(v);
    if (wl_lane() < LR) Row::store(sh.lbl, W, v);
    __syncwarp();
  }
  __device__ void label_one(int a) {
    uint32_t v[KW];
    Row::load(g.exp_term + (size_t)a * W, W, v);
    if (wl_lane() < LR) Row::store(sh.lbl, W, v);
    __syncwarp();
  }

  // a node built from labelled / epsilon arrivals, closed and stored
  __device__ bool simple_column(int& c_out, int src, bool eps, bool gap) {
    int c = open_column();
    if (c < 0) return false;
    arrive(src, !eps);
    close_column(c, gap);
    finish_column(c);
    c_out = c;
    return status == 0;
  }

  // ------------------------------------------------------------ span step
  __device__ static uint32_t tail_word(const LexEntry& e, int i) {
    uint32_t v = 0;
    for (int j = 0; j < 4; ++j) {
      int t = 1 + 4 * i + j;
      v |= (uint32_t)(t < e.len ? e.term[t] : 0) << (8 * j);
    }
    return v;
  }

  __device__ EPIC_STEP bool span_step(int tok) {
    if (g.lazy.stats && wl_lane() == 0) atomicAdd(&g.lazy.stats[0], (unsigned long long)nf);
    int ng = 0;
    PH_BEGIN(t_group);
    // grouping, 32 frontier elements at a time
    for (int base = 0; base < nf; base += 32) {
      int f = base + (int)wl_lane();
      bool live = false;
      LexEntry e;
      int src = -1;
      if (f < nf) {
        e = lex_at(g, table, tok, ws.f_q[f]);
        src = ws.f_c[f];
        live = e.end != 0xFFFF;
      }
      uint32_t t0 = live ? tail_word(e, 0) : 0, t1 = live ? tail_word(e, 1) : 0, t2 = live ? tail_word(e, 2) : 0;
      int gid = -1;
      if (live) {
        for (int gi = 0; gi < ng; ++gi) {
          if (ws.g_src[gi] == src && ws.g_end[gi] == e.end && ws.g_len[gi] == e.len &&
              ws.g_tail[gi * 4] == t0 && ws.g_tail[gi * 4 + 1] == t1 && ws.g_tail[gi * 4 + 2] == t2) {
            gid = gi;
            break;
          }
        }
      }
      unsigned pending = __ballot_sync(0xffffffffu, live && gid < 0);
      while (pending) {
        int l = __ffs(pending) - 1;
        int ksrc = __shfl_sync(0xffffffffu, src, l);
        int kend = __shfl_sync(0xffffffffu, (int)(live ? e.end : 0), l);
        int klen = __shfl_sync(0xffffffffu, (int)(live ? e.len : 0), l);
        uint32_t k0 = __shfl_sync(0xffffffffu, t0, l), k1 = __shfl_sync(0xffffffffu, t1, l),
                 k2 = __shfl_sync(0xffffffffu, t2, l);
        if (ng >= kWMaxQ) {
          status = 1;
          return false;
        }
        if (wl_lane() == 0) {
          ws.g_src[ng] = ksrc;
          ws.g_end[ng] = kend;
          ws.g_len[ng] = klen;
          ws.g_tail[ng * 4] = k0;
          ws.g_tail[ng * 4 + 1] = k1;
          ws.g_tail[ng * 4 + 2] = k2;
          for (int w = 0; w < 8; ++w) ws.g_lbl[ng * 8 + w] = 0;
        }
        __syncwarp();
        bool same = live && gid < 0 && src == ksrc && (int)e.end == kend && (int)e.len == klen && t0 == k0 &&
                    t1 == k1 && t2 == k2;
        if (same) gid = ng;
        pending &= ~__ballot_sync(0xffffffffu, same);
        ++ng;
      }
      if (live && e.len > 0) atomicOr(&ws.g_lbl[gid * 8 + (e.term[0] >> 5)], 1u << (e.term[0] & 31));
      __syncwarp();
    }
    PH_END(0, t_group);
    // intermediate nodes: the run up to its last terminal; groups with the
    // same source, first-terminal set and terminals before the last one
    // spell the same paths up to it, so they share one chain of nodes
    for (int gi = 0; gi < ng; ++gi) {
      int len = ws.g_len[gi];
      int cur = ws.g_src[gi];
      if (len >= 2) {
        int share = -1;
        for (int gb = 0; gb < gi && share < 0; gb += 32) {
          const int gj = gb + (int)wl_lane();
          bool same = gj < gi && ws.g_len[gj] == len && ws.g_src[gj] == cur;
          for (int w = 0; w < 8 && same; ++w) same = ws.g_lbl[gj * 8 + w] == ws.g_lbl[gi * 8 + w];
          for (int t = 1; t + 1 < len && same; ++t) same = tail_term(gj, t) == tail_term(gi, t);
          const unsigned m = __ballot_sync(0xffffffffu, same);
          if (m) share = gb + __ffs(m) - 1;
        }
        if (share >= 0) {
          if (wl_lane() == 0) ws.g_last[gi] = ws.g_last[share];
          __syncwarp();
          continue;
        }
      }
      for (int t = 0; t + 1 < len; ++t) {
        if (t == 0) {
          label_set(ws.g_lbl + gi * 8);
        } else {
          uint32_t tw = ws.g_tail[gi * 4 + ((t - 1) >> 2)];
          label_one((tw >> (8 * ((t - 1) & 3))) & 0xff);
        }
        int c;
        if (!simple_column(c, cur, false, false)) return false;
        cur = c;
      }
      if (wl_lane() == 0) ws.g_last[gi] = cur;
      __syncwarp();
    }
    // the distinct end states, ascending (the old frontier is consumed)
    int nt = 0;
    int prev = -1;
    for (;;) {
      int best = 0x7fffffff;
      for (int gi = wl_lane(); gi < ng; gi += 32) {
        int e = ws.g_end[gi];
        if (e > prev && e < best) best = e;
      }
      for (int off = 16; off; off >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, off));
      if (best == 0x7fffffff) break;
      if (wl_lane() == 0) ws.f_q[nt] = best;
      ++nt;
      prev = best;
    }
    __syncwarp();
    // end nodes with the same arrivals (sources and labels) have the same
    // incoming paths: one column serves all their lexer states; the smallest
    // equal end is the representative (ws.f_c holds a hash of the arrivals
    // until the columns are made)
    for (int ti = wl_lane(); ti < nt; ti += 32) ws.f_c[ti] = (int32_t)arrivals_hash(ws.f_q[ti], ng);
    __syncwarp();
    for (int ti = wl_lane(); ti < nt; ti += 32) {
      int rep = ti;
      for (int tj = 0; tj < ti; ++tj)
        if (ws.f_c[tj] == ws.f_c[ti] && same_arrivals(ws.f_q[ti], ws.f_q[tj], ng)) {
          rep = tj;
          break;
        }
      ws.key_q[ti] = rep;
    }
    __syncwarp();
    for (int ti = 0; ti < nt; ++ti) {
      if (ws.key_q[ti] != ti) continue;
      const int best = ws.f_q[ti];
      int c = open_column();
      if (c < 0) return false;
      for (int gi = 0; gi < ng; ++gi) {
        if (ws.g_end[gi] != best) continue;
        int len = ws.g_len[gi];
        if (len == 0) {
          arrive(ws.g_src[gi], false);
        } else if (len == 1) {
          label_set(ws.g_lbl + gi * 8);
          arrive(ws.g_src[gi], true);
        } else {
          label_one(tail_term(gi, len - 1));
          arrive(ws.g_last[gi], true);
        }
      }
      bool defer = false;
      if (EXT && defer_to_gap) {
        bool all_eps = true;
        for (int tj = (int)wl_lane(); tj < nt; tj += 32)
          if (ws.key_q[tj] == ti && !eps_into_gap(ws.f_q[tj])) all_eps = false;
        defer = __all_sync(0xffffffffu, all_eps);
      }
      if (!defer) close_column(c, false);  // else: rows as they arrived
      finish_column(c);
      if (status) return false;
      if (wl_lane() == 0) ws.f_c[ti] = c;
      __syncwarp();
    }
    // the new frontier: (end state, column) of the non-empty columns
    for (int ti = wl_lane(); ti < nt; ti += 32)
      if (ws.key_q[ti] != ti) ws.f_c[ti] = ws.f_c[ws.key_q[ti]];  // representatives are columns by now
    __syncwarp();
    int nk = 0;
    for (int ti = 0; ti < nt; ++ti) {
      const int c = ws.f_c[ti];
      if (column_empty(c)) continue;
      if (wl_lane() == 0) {
        ws.f_q[nk] = ws.f_q[ti];
        ws.f_c[nk] = c;
      }
      __syncwarp();
      ++nk;
    }
    nf = nk;
    return true;
  }

  // terminal t (1 .. len-1) of group gi's run
  __device__ int tail_term(int gi, int t) const {
    return (ws.g_tail[gi * 4 + ((t - 1) >> 2)] >> (8 * ((t - 1) & 3))) & 0xff;
  }
  // arrival of group gi into its end node: source column and label set (all
  // zero: epsilon)
  __device__ int arrival_src(int gi) const { return ws.g_len[gi] >= 2 ? ws.g_last[gi] : ws.g_src[gi]; }
  __device__ uint32_t arrival_lbl(int gi, int w) const {
    const int len = ws.g_len[gi];
    if (len == 0) return 0u;
    if (len == 1) return ws.g_lbl[gi * 8 + w];
    const int a = tail_term(gi, len - 1);
    return (w == (a >> 5)) ? (1u << (a & 31)) : 0u;
  }
  __device__ uint32_t arrivals_hash(int e, int ng) const {
    uint32_t h = 0;
    for (int gi = 0; gi < ng; ++gi) {
      if (ws.g_end[gi] != e) continue;
      uint32_t x = (uint32_t)arrival_src(gi) * 0x9E3779B1u + (ws.g_len[gi] == 0 ? 0x85EBCA6Bu : 0u);
      for (int w = 0; w < 8; ++w) x = (x ^ arrival_lbl(gi, w)) * 0xC2B2AE35u + (uint32_t)w;
      h += x ^ (x >> 16);
    }
    return h;
  }
  // do end states e1 and e2 receive the same arrivals?  (one lane)
  __device__ bool same_arrivals(int e1, int e2, int ng) const {
    int n1 = 0, n2 = 0;
    for (int gi = 0; gi < ng; ++gi) {
      n1 += ws.g_end[gi] == e1;
      n2 += ws.g_end[gi] == e2;
    }
    if (n1 != n2) return false;
    for (int gi = 0; gi < ng; ++gi) {
      if (ws.g_end[gi] != e1) continue;
      bool found = false;
      for (int gj = 0; gj < ng && !found; ++gj) {
        if (ws.g_end[gj] != e2 || arrival_src(gj) != arrival_src(gi)) continue;
        bool same = (ws.g_len[gi] == 0) == (ws.g_len[gj] == 0);
        for (int w = 0; w < 8; ++w) same &= arrival_lbl(gi, w) == arrival_lbl(gj, w);
        found = same;
      }
      if (!found) return false;
    }
    return true;
  }

  // ------------------------------------------------------------ the walk
  __device__ static int token_at(const int32_t* x, int sp, int st, int i) { return i == sp ? st : x[i]; }

  // x (+) {(sp, st)}; returns 1 valid, 0 invalid, -1 overflow, -2 bad input
  __device__ int run(const int32_t* x, int n, int sp, int st) {
    ncols = base_cols;
    nent = 0;
    status = 0;
    nf = 0;
    if (wl_lane() == 0) ws.col_off[0] = 0;
    __syncwarp();
    if (sp >= 0 && (sp >= n || x[sp] >= 0 || st < 0 || st >= vocab)) return -2;
    int r = run_inner(x, n, sp, st);
    if (r < 0 || status) {
      cleanup();
      return status == 1 ? -1 : (r < 0 ? r : -1);
    }
    return r;
  }

  // Arrivals of the frontier into the open column: by an epsilon edge, by the
  // pending lexeme's terminal, or none (a dead end); frontier elements with
  // the same column and the same edge arrive once.  At a gap a pending lexeme
  // some byte can extend stays open (epsilon), one no byte can extend emits
  // its terminal; at the END the pending lexeme is flushed.
  __device__ void arrive_frontier(bool gap) {
    for (int f = wl_lane(); f < nf; f += 32) {
      const int q = ws.f_q[f], a = g.dfa_accept[q];
      int kind = -2;
      if (q == 0 || (gap && g.dfa_ext[q]) || (a >= 0 && g.skip[a]))
        kind = -1;
      else if (a >= 0)
        kind = a;
      ws.g_len[f] = kind;
    }
    __syncwarp();
    for (int f = 0; f < nf; ++f) {
      const int kind = ws.g_len[f], c = ws.f_c[f];
      if (kind == -2) continue;
      bool dup = false;
      for (int h = wl_lane(); h < f; h += 32) dup |= ws.f_c[h] == c && ws.g_len[h] == kind;
      if (__any_sync(0xffffffffu, dup)) continue;
      if (kind >= 0) label_one(kind);
      arrive(c, kind >= 0);
    }
  }
  __device__ int gap_from_frontier() {
    int c = open_column();
    if (c >= 0) arrive_frontier(true);
    return c;
  }
  __device__ int end_from_frontier() {
    int c = open_column();
    if (c >= 0) arrive_frontier(false);
    return c;
  }
  // frontier of a span that starts at column src: q0 at the sequence start,
  // every lexer state after a gap
  __device__ void frontier_from(int src, bool at_begin) {
    if (at_begin) {
      if (wl_lane() == 0) {
        ws.f_q[0] = 0;
        ws.f_c[0] = src;
      }
      nf = 1;
    } else {
      for (int q = wl_lane(); q < g.Q; q += 32) {
        ws.f_q[q] = q;
        ws.f_c[q] = src;
      }
      nf = g.Q;
    }
    __syncwarp();
  }
  __device__ int run_inner(const int32_t* x, int n, int sp, int stok) {
    int i = 0;
    bool first = true;
    int prev_gap = -1;
    while (i < n) {
      int t0 = token_at(x, sp, stok, i);
      int j = i;
      if (t0 < 0) {
        while (j < n && token_at(x, sp, stok, j) < 0) ++j;
        int c;
        if (first) {
          c = open_column();
          if (c < 0) return -1;
          start_col = c;
          seed(c);
        } else {
          c = gap_from_frontier();
          if (c < 0) return -1;
        }
        close_column(c, true);
        finish_column(c);
        if (status) return -1;
        prev_gap = c;
        if (column_empty(c)) return 0;
      } else {
        while (j < n && token_at(x, sp, stok, j) >= 0) ++j;
        int src;
        if (first) {
          int c = open_column();
          if (c < 0) return -1;
          start_col = c;
          seed(c);
          close_column(c, false);
          finish_column(c);
          if (status) return -1;
          src = c;
        } else {
          src = prev_gap;
        }
        frontier_from(src, first);
        for (int p = i; p < j && nf > 0; ++p) {
          int tok = token_at(x, sp, stok, p);
          if (tok < 0 || tok >= vocab) return -2;
          if (!span_step(tok)) return -1;
        }
        if (nf == 0) return 0;
        if (j == n) {  // END: flush the pending lexeme
          int c = end_from_frontier();
          if (c < 0) return -1;
          close_column(c, false);
          finish_column(c);
          if (status) return -1;
          return accepts(c, start_col) ? 1 : 0;
        }
      }
      first = false;
      i = j;
    }
    return accepts(prev_gap, start_col) ? 1 : 0;
  }
};

}  // namespace epic
