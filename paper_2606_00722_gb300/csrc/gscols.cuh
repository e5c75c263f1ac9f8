// Earley columns of the CTA walks: one CTA closes each column of a chart, its
// warps working through the column's origins on their own (Alg. 3's
// completion).
//
// Completing nonterminal A from origin o at column c advances the items of
// column o that wait on A; those items have origins o2 <= o, so a row with
// origin o only receives from origins >= o.  The sweep therefore runs from
// the highest origin down, asynchronously: each warp repeatedly claims the
// highest dirty origin below c (clearing its bit), closes its row together
// with the self-loop through the entry of column o with origin o (the items
// predicted at o) in registers, and scatters the nonterminals that no earlier
// visit completed over the other entries of column o with atomic ORs, marking
// the rows it changes dirty again.  A row may be claimed while another warp
// still writes into it; the writer sets the dirty bit after its writes
// (fenced), so the row is visited again and nothing is lost.  The sweep ends
// when no bit is dirty and no warp holds an origin.  The rules are monotone,
// so the result is the least fixpoint whatever the order.
//
// What bounds it: the chain of dependent visits, each a few dependent
// shared-memory steps long, and the loads of column o's entries.  Hence
//  - the rows of the open column, their completed-nonterminal sets, the column
//    offsets and the span step's tables live in shared memory (an origin gets
//    a row slot on first touch; a column with more origins than slots puts the
//    rest in the global stage).  A visit makes no global store, and its fences
//    wait for shared memory only;
//  - completed nonterminals are read off a row by one lane per nonterminal
//    testing its (word, mask) pairs, 32 nonterminals per ballot, and the items
//    waiting on new nonterminals are OR-ed from EXP_NT rows: no per-item loops
//    and no shared-memory atomics;
//  - a row takes LR lanes of KW consecutive words (rows are padded to a
//    multiple of four words, so a lane moves 16 bytes at a time and a shift by
//    one item costs one shuffle): 4 lanes x 4 words up to 16 words, 16 x 4 up
//    to 64, 32 x 8 up to 256.  A warp scatters 32 / LR entries per step, and
//    when it works on one row its lane groups hold copies and share out the
//    EXP_NT rows.  (With one word per lane and 32-word steps a 64-word row took
//    about 70 instructions per scattered entry; issue is what bounds a sweep
//    with four warps per scheduler.)
//  - all nonterminals that complete at c from o through chains at the self
//    entry (B -> A, or at gaps any production around A) follow from the
//    directly completed ones by a table, so a visit is one pass instead of a
//    round per link (2.7 on average for clike-512).
// Predictions at c only feed row c (items predicted at c have origin c), and
// the prediction closures are closed under further predictions, so they are
// made once, after the lower origins are closed; completions from c at c are
// the nullable / gap advances of every row (Aycock & Horspool; inside a gap
// every symbol derives some terminal string of the trimmed grammar).
#pragma once
#include "rows.cuh"
#include "walk.cuh"
#include "warpwalk.cuh"  // phase timers

namespace epic {

constexpr int kGsMaxWarps = 16;
// Threads of a CTA walk (128 registers each).  Sixteen warps; eight for narrow
// rows when there are more walks than SMs, so that two CTAs share one (512
// threads at 64 registers spilled: smiles-256 forward charts 95 ms against 68);
// four for tiny grammars, whose columns hold too few origins for more.  With
// one narrow walk per SM sixteen warps are the faster: smiles 48 x 144 exact
// tests 20.5 -> 15.8 ms.
inline int gs_sms() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}
inline int gs_threads(int W, long long walks, int sms) {
  return W <= 4 ? 128 : (W <= 16 && walks > sms ? 256 : 32 * kGsMaxWarps);
}
constexpr long long kGsMaxSteps = 1ll << 22;  // origin visits per column and warp
constexpr long long kGsMaxIdle = 1ll << 24;   // polls of an idle warp per column

// Grammar masks of W words, staged in shared memory.
struct GsTables {
  const uint32_t* complete;
  const uint32_t* any_nt;
  const uint32_t* adv_pow;  // [2][steps][W] (DevGrammar::adv_pow)
};

__host__ __device__ inline size_t gs_tables_bytes(int W, int steps) {
  auto r = [](size_t b) { return (b + 15) & ~(size_t)15; };
  return 2 * r((size_t)W * 4) + r((size_t)2 * steps * W * 4);
}

// Block: copy the tables into smem (gs_tables_bytes) and point t at them.
__device__ inline void gs_stage_tables(const DevGrammar& g, unsigned char* smem, GsTables& t) {
  unsigned char* p = smem;
  auto put = [&](const void* src, size_t bytes) -> void* {
    void* dst = p;
    const uint16_t* s2 = (const uint16_t*)src;
    uint16_t* d2 = (uint16_t*)dst;
    for (size_t i = threadIdx.x; i < bytes / 2; i += blockDim.x) d2[i] = s2[i];
    p += (bytes + 15) & ~(size_t)15;
    return dst;
  };
  t.complete = (const uint32_t*)put(g.complete, (size_t)g.W * 4);
  t.any_nt = (const uint32_t*)put(g.any_nt, (size_t)g.W * 4);
  t.adv_pow = (const uint32_t*)put(g.adv_pow, (size_t)2 * g.adv_steps * g.W * 4);
  __syncthreads();
}

// Dynamic shared memory of the CTA walks (byte offsets): WalkSmem, the tables
// above, then the pieces below; `rows` row slots take what is left.
struct GsPlan {
  uint32_t o_w4, o_m4;     // complete items by nonterminal (DevGrammar::cpl4w, cpl4m) ...
  uint32_t o_off, o_list;  // ... and as lists
  uint32_t o_woff, o_wait; // items waiting on each nonterminal, as lists; 0: read from global memory
  uint32_t o_scr;          // per-warp scratch, W words each
  uint32_t o_col;          // column offsets [nmax + 1]
  uint32_t o_slot;         // row slot of each origin [nmax] (uint16)
  uint32_t o_self;         // bit o: column o has an entry with origin o
  uint32_t o_gap;          // bit o: column o is a gap
  uint32_t o_fol;          // DevGrammar::follow; 0: read from global memory
  uint32_t o_exp;          // EXP_NT rows; 0: read from global memory
  uint32_t o_next;         // DevGrammar::next_t (wide rows); 0: read from global memory
  uint32_t o_walk;         // span step tables; 0: in the global workspace
  uint32_t o_zero;         // a row of zeros, for origins without a slot
  uint32_t o_rows, o_done; // row slots, completed nonterminals per slot
  int rows;
  uint32_t bytes;
};

constexpr uint32_t kSlotNone = 0xFFFFu, kSlotGlobal = 0xFFFEu;
constexpr size_t kGsWalkBytesPerState = 7 * 4 + 16 + 32 + 16;  // WalkScratch per lexer state

// limit: dynamic shared memory a CTA may take.  Narrow rows keep to what lets
// two CTAs share an SM.
inline GsPlan gs_plan(const DevGrammar& g, int nmax, size_t limit) {
  auto r = [](size_t b) { return (b + 15) & ~(size_t)15; };
  GsPlan p;
  size_t o = kWalkSmemBytes + r(gs_tables_bytes(g.W, g.adv_steps));
  auto put = [&](size_t bytes) {
    const size_t at = o;
    o += r(bytes);
    return (uint32_t)at;
  };
  p.o_w4 = put((size_t)g.V * 8);
  p.o_m4 = put((size_t)g.V * 16);
  p.o_off = put((size_t)(g.V + 1) * 4);
  p.o_list = put((size_t)g.n_cpl * 8);
  const bool wait_in = (size_t)g.n_wait * 8 <= 12 * 1024;
  p.o_woff = wait_in ? put((size_t)(g.V + 1) * 4) : 0;
  p.o_wait = wait_in ? put((size_t)g.n_wait * 8) : 0;
  p.o_scr = put((size_t)kGsMaxWarps * g.W * 4);
  p.o_col = put((size_t)(nmax + 1) * 4);
  p.o_slot = put((size_t)nmax * 2);
  p.o_self = put((size_t)((nmax + 31) / 32) * 4);
  p.o_gap = put((size_t)((nmax + 31) / 32) * 4);
  p.o_zero = put((size_t)g.W * 4);
  const size_t per_row = (size_t)(g.W + g.VW) * 4;
  const size_t least = 64 * per_row;  // rows that always come first
  const size_t walk = (size_t)g.Q * kGsWalkBytesPerState, ex = (size_t)g.V * g.W * 4;
  p.o_walk = o + r(walk) + least <= limit ? put(walk) : 0;
  const size_t fol = (size_t)4 * g.V * g.VW * 4;
  p.o_fol = fol <= 16 * 1024 && o + r(fol) + least <= limit ? put(fol) : 0;
  const size_t nx = (size_t)64 * g.W;
  p.o_next = g.W > 64 && o + r(nx) + least <= limit ? put(nx) : 0;
  p.o_exp = o + r(ex) + 2 * least <= limit ? put(ex) : 0;
  const size_t left = limit > o + 32 ? limit - o - 32 : 0;
  long long rows = (long long)(left / per_row);
  rows = rows > nmax ? nmax : rows;
  rows = rows > 1024 ? 1024 : rows;
  p.rows = (int)rows;
  p.o_rows = put((size_t)rows * g.W * 4);
  p.o_done = put((size_t)rows * g.VW * 4);
  p.bytes = (uint32_t)o;
  return p;
}
// 227 KB per CTA less the static shared memory of the walk kernels (at most
// 10 KB); half of an SM's 228 KB for the narrow rows
inline size_t gs_limit(int W) { return W <= 16 ? (size_t)102 * 1024 : (size_t)216 * 1024; }

// The steps of one column are calls (not inlined at each of the walk's many
// uses): inlined, the selection kernels took six minutes to compile.
template <bool REC, class S>
class EarleyColsGS {
 public:
  static constexpr int KW = S::KW, LR = S::LR, NG = S::NG;
  using Row = RowRegs<S>;
  static constexpr bool kRecord = REC;
  const DevGrammar& g;
  const GsTables& tb;
  const GsPlan& plan;
  Workspace ws;  // col_off is the shared-memory copy
  WsDims dims;
  int W, VW, R;
  const BlockRec* rec = nullptr;
  uint32_t *rows, *done, *selfb, *gapb;
  uint16_t* slot_of;

  // What the visits and scatters of a column read at every step, copied to
  // registers once per call: the object itself lies in local memory, and its
  // members would be read again after every barrier and atomic.
  struct Hot {
    int W, VW, V, R, steps, nullable;
    uint32_t s_rows, s_zero;      // shared addresses: row slots, the zero row
    const uint32_t *adv, *complete, *selfb, *gapb, *exp_nt, *follow;
    uint32_t *scr, *rows, *done, *stage, *bdone;
    uint16_t* slot_of;
    const int32_t *c_off, *col, *org;
    const int16_t* next_t;
    const uint2 *c_lst, *w4;
    const uint4* m4;
    const uint32_t* bits;
    __device__ __forceinline__ uint32_t slot(int o) const { return *(const volatile uint16_t*)(slot_of + o); }
    __device__ __forceinline__ uint32_t* done_of(uint32_t s, int o) const {
      return s < (uint32_t)R ? done + (size_t)s * VW : bdone + (size_t)o * VW;
    }
  };
  __device__ __forceinline__ Hot hot() const {
    unsigned char* m = gs_smem();
    Hot h;
    h.W = W;
    h.VW = VW;
    h.V = g.V;
    h.R = R;
    h.steps = g.adv_steps;
    h.nullable = g.any_nullable;
    h.s_rows = gs_saddr(m + plan.o_rows);
    h.s_zero = gs_saddr(m + plan.o_zero);
    h.adv = tb.adv_pow;
    h.complete = tb.complete;
    h.selfb = (const uint32_t*)(m + plan.o_self);
    h.gapb = (const uint32_t*)(m + plan.o_gap);
    h.follow = plan.o_fol ? (const uint32_t*)(m + plan.o_fol) : g.follow;
    h.next_t = plan.o_next ? (const int16_t*)(m + plan.o_next) : g.next_t;
    h.exp_nt = plan.o_exp ? (const uint32_t*)(m + plan.o_exp) : g.exp_nt;
    h.scr = (uint32_t*)(m + plan.o_scr) + (size_t)(threadIdx.x >> 5) * W;
    h.rows = (uint32_t*)(m + plan.o_rows);
    h.done = (uint32_t*)(m + plan.o_done);
    h.stage = ws.stage;
    h.bdone = ws.bdone;
    h.slot_of = (uint16_t*)(m + plan.o_slot);
    h.w4 = (const uint2*)(m + plan.o_w4);
    h.m4 = (const uint4*)(m + plan.o_m4);
    h.c_off = (const int32_t*)(m + plan.o_off);
    h.c_lst = (const uint2*)(m + plan.o_list);
    h.col = (const int32_t*)(m + plan.o_col);
    h.org = ws.org;
    h.bits = ws.bits;
    return h;
  }

  __device__ EarleyColsGS(const DevGrammar& g_, const GsTables& t_, const GsPlan& p, unsigned char* smem, Workspace w,
                          WsDims d)
      : g(g_), tb(t_), plan(p), ws(w), dims(d), W(g_.W), VW(g_.VW), R(p.rows) {
    ws.col_off = (int32_t*)(smem + p.o_col);
    slot_of = (uint16_t*)(smem + p.o_slot);
    selfb = (uint32_t*)(smem + p.o_self);
    gapb = (uint32_t*)(smem + p.o_gap);
    rows = (uint32_t*)(smem + p.o_rows);
    done = (uint32_t*)(smem + p.o_done);
  }

  // The walk's span tables in shared memory when they fit.
  __device__ static void place_scratch(const DevGrammar& g, const GsPlan& p, unsigned char* smem, WalkScratch& sc) {
    if (!p.o_walk) return;
    unsigned char* q = smem + p.o_walk;
    const size_t Q = (size_t)g.Q;
    sc.ent = (LexEntry*)q;
    q += Q * 16;
    sc.g_tail = (uint8_t*)q;
    q += Q * 16;
    sc.g_lbl = (uint32_t*)q;
    q += Q * 32;
    int32_t** a[7] = {&sc.g_src, &sc.g_end, &sc.g_len, &sc.g_last, &sc.f_q, &sc.f_c, &sc.key_q};
    for (int i = 0; i < 7; ++i, q += Q * 4) *a[i] = (int32_t*)q;
  }

  // Block, once per kernel: the shared tables, empty slots, zero rows.
  __device__ void init(unsigned char* smem) {
    for (int v = threadIdx.x; v < g.V; v += blockDim.x) {
      ((uint2*)(smem + plan.o_w4))[v] = g.cpl4w[v];
      ((uint4*)(smem + plan.o_m4))[v] = g.cpl4m[v];
    }
    for (int v = threadIdx.x; v <= g.V; v += blockDim.x) ((int32_t*)(smem + plan.o_off))[v] = g.cpl_off[v];
    for (int i = threadIdx.x; i < g.n_cpl; i += blockDim.x) ((uint2*)(smem + plan.o_list))[i] = g.cpl[i];
    if (plan.o_wait) {
      for (int v = threadIdx.x; v <= g.V; v += blockDim.x) ((int32_t*)(smem + plan.o_woff))[v] = g.wait_off[v];
      for (int i = threadIdx.x; i < g.n_wait; i += blockDim.x) ((uint2*)(smem + plan.o_wait))[i] = g.wait[i];
    }
    if (plan.o_exp) {
      uint32_t* ex = (uint32_t*)(smem + plan.o_exp);
      for (int i = threadIdx.x; i < g.V * W; i += blockDim.x) ex[i] = g.exp_nt[i];
    }
    if (plan.o_next) {
      int16_t* t = (int16_t*)(smem + plan.o_next);
      for (int i = threadIdx.x; i < 32 * W; i += blockDim.x) t[i] = g.next_t[i];
    }
    if (plan.o_fol) {
      uint32_t* f = (uint32_t*)(smem + plan.o_fol);
      for (int i = threadIdx.x; i < 4 * g.V * VW; i += blockDim.x) f[i] = g.follow[i];
    }
    for (int i = threadIdx.x; i < W; i += blockDim.x) ((uint32_t*)(smem + plan.o_zero))[i] = 0;
    for (int i = threadIdx.x; i < R * W; i += blockDim.x) rows[i] = 0;
    for (int i = threadIdx.x; i < R * VW; i += blockDim.x) done[i] = 0;
    for (int i = threadIdx.x; i < dims.nmax; i += blockDim.x) slot_of[i] = (uint16_t)kSlotNone;
    __syncthreads();
  }

  __device__ int nwarps() const { return blockDim.x >> 5; }
  __device__ bool column_has_accept(int c, int start_col) { return accepts(c, start_col); }
  __device__ void arrive_labels(int src, bool eps) { arrive(src, !eps); }

  __device__ void reset() {
    if (threadIdx.x == 0) {
      walk_sh().ncols = 0;
      walk_sh().nent = 0;
      walk_sh().status = kWalkOk;
      walk_sh().nedges = 0;
      ws.col_off[0] = 0;
      walk_gs().labelled = 0;
      walk_gs().nslots = 0;
    }
    clear_bitmap(walk_sh().touched, kMaxCols);
    clear_bitmap(walk_sh().dirty, kMaxCols);
    clear_bitmap(selfb, dims.nmax);
    clear_bitmap(gapb, dims.nmax);
    __syncthreads();
  }

  __device__ int ncols() const { return walk_sh().ncols; }
  // The next column, or -1 when there is no room (known to every thread: the
  // status is not written here, slower warps may still read it for the column
  // before).
  __device__ int open_column() {
    const int c = walk_sh().ncols;
    return c < dims.nmax && c < kMaxCols ? c : -1;
  }

  // ------------------------------------------------------------ row slots
  __device__ __forceinline__ static uint32_t vld(const uint32_t* p) { return *(const volatile uint32_t*)p; }
  __device__ __forceinline__ uint32_t slot(int o) const { return *(const volatile uint16_t*)(slot_of + o); }
  __device__ __forceinline__ uint32_t* row_of(uint32_t s, int o) const {
    return s < (uint32_t)R ? rows + (size_t)s * W : ws.stage + (size_t)o * W;
  }
  __device__ __forceinline__ uint32_t* done_of(uint32_t s, int o) const {
    return s < (uint32_t)R ? done + (size_t)s * VW : ws.bdone + (size_t)o * VW;
  }
  // One thread: the slot of origin o, claimed on its first touch.  A claim
  // that loses the race leaves its slot unused (zero) in this column.
  __device__ __forceinline__ uint32_t claim(int o) { return claim(slot_of, R, o); }
  __device__ static uint32_t claim(uint16_t* slot_of, int R, int o) {
    uint32_t s = *(const volatile uint16_t*)(slot_of + o);
    if (s != kSlotNone) return s;
    const int t = atomicAdd(&walk_gs().nslots, 1);
    const uint32_t want = t < R ? (uint32_t)t : kSlotGlobal;
    const unsigned short old =
        atomicCAS((unsigned short*)(slot_of + o), (unsigned short)kSlotNone, (unsigned short)want);
    return old == (unsigned short)kSlotNone ? want : (uint32_t)old;
  }
  __device__ static __forceinline__ void mark(int o) {
    atomicOr(&walk_sh().touched[o >> 5], 1u << (o & 31));
    atomicOr(&walk_sh().dirty[o >> 5], 1u << (o & 31));
  }

  // ------------------------------------------------------------ row kernels
  // Warp: row(origin) |= bits & m, shifted to the next item when SHIFT, for
  // entries of kb .. ke - 1; marks the origins whose rows change.  Entries go
  // NG at a time, steps first, first + stride, ...; m: the mask words of this
  // lane.  Origins and row addresses of 32 entries are looked up at once; the
  // common case (the row already holds the items) is loads, a shuffle and a
  // vote.
  template <bool SHIFT>
  __device__ static __forceinline__ void scatter(const Hot& h, int kb, int ke, const uint32_t (&m)[KW], int first, int stride) {
    constexpr int U = LR == 16 ? 4 : 2;  // steps in flight
    const int lane = threadIdx.x & 31, li = Row::li(), gi = Row::gi();
    const int ne = ke - kb;
    const int W = h.W, R = h.R;
    const uint32_t* bits = h.bits + (size_t)kb * W;
    const uint32_t s_rows = h.s_rows, s_zero = h.s_zero;
    const unsigned group = LR == 32 ? 0xffffffffu : ((1u << LR) - 1u) << (gi * LR);
    for (int c0 = 0; (c0 * stride + first) * NG < ne; c0 += LR) {
      // lane t looks up entry t of the chunk: step c0 + t / NG, place t % NG
      const int et = ((c0 + lane / NG) * stride + first) * NG + lane % NG;
      const bool okt = et < ne;
      const int o_t = okt ? h.org[kb + et] : 0;
      const uint32_t s_t = okt ? h.slot(o_t) : kSlotNone;
      const uint32_t a_t = s_t < (uint32_t)R ? s_rows + s_t * (uint32_t)(W * 4) : s_zero;
      const int steps = min(LR, (ne - first * NG + stride * NG - 1) / (stride * NG) - c0);
      const int last_t = 31 - __clz(__ballot_sync(0xffffffffu, okt));  // the lane of the chunk's last entry
      for (int u0 = 0; u0 < steps; u0 += U) {
        uint32_t v[U][KW];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if constexpr (LR == 4) {  // eight entries a step: columns often end within it
            const int e = ((c0 + u0 + u) * stride + first) * NG + gi;
            if (u0 + u < steps && e < ne) {
              Row::load(bits + (size_t)e * W, W, v[u]);
            } else {
#pragma unroll
              for (int i = 0; i < KW; ++i) v[u][i] = 0u;
            }
          } else {  // past the end: the last entry again
            Row::load_any(bits + (size_t)min(((c0 + min(u0 + u, steps - 1)) * stride + first) * NG + gi, ne - 1) * W, W,
                          v[u]);
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          // (its lookup is in lane t of this chunk)
          const int t = LR == 4 ? ((u0 + u) * NG + gi) & 31 : min(min(u0 + u, steps - 1) * NG + gi, last_t);
          const uint32_t addr = __shfl_sync(0xffffffffu, a_t, t);
          uint32_t q[KW];
          if constexpr (LR == 4)
            Row::load_shared(addr, W, q);
          else
            Row::load_shared_any(addr, W, q);
#pragma unroll
          for (int i = 0; i < KW; ++i) v[u][i] &= m[i];
          if (SHIFT) Row::shift_up(v[u]);
          uint32_t nw = 0;
#pragma unroll
          for (int i = 0; i < KW; ++i) nw |= v[u][i] & ~q[i];
          const unsigned bal = __ballot_sync(0xffffffffu, nw != 0);
          if (bal) {
            const bool mine = (bal & group) != 0;
            const int o2 = __shfl_sync(0xffffffffu, o_t, t);
            uint32_t s = __shfl_sync(0xffffffffu, s_t, t);
            if (mine && li == 0 && s == kSlotNone) s = claim(h.slot_of, R, o2);
            s = __shfl_sync(0xffffffffu, s, 0, LR);
            bool ch = mine;
            if (mine && s < (uint32_t)R) {
              const uint32_t d = s_rows + s * (uint32_t)(W * 4) + (uint32_t)(li * KW) * 4u;
#pragma unroll
              for (int i = 0; i < KW; ++i)
                if (v[u][i] & ~q[i]) gs_red_or(d + 4u * i, v[u][i]);
            } else if (mine) {  // no slot left: the row is in the global stage
              uint32_t* d = h.stage + (size_t)o2 * W + li * KW;
              ch = false;
#pragma unroll
              for (int i = 0; i < KW; ++i)
                if (v[u][i] && (v[u][i] & ~vld(d + i))) {
                  atomicOr(d + i, v[u][i]);
                  ch = true;
                }
            }
            __threadfence_block();  // every lane's row writes before the dirty bit
            const unsigned chm = __ballot_sync(0xffffffffu, ch);
            if (li == 0 && (chm & group)) mark(o2);
          }
        }
      }
    }
    __syncwarp();
  }

  // Arrivals: for every entry (o, y) of column src, row(o) |= shift(y & lbl)
  // (labelled) or row(o) |= y (epsilon).
  __device__ __noinline__ void arrive(int src, bool shift) {
    const int warp = threadIdx.x >> 5, nw = nwarps();
    if (shift && threadIdx.x == 0) walk_gs().labelled = 1;
    if (REC && threadIdx.x == 0) {
      if (walk_sh().nedges >= rec->edge_cap) {
        walk_sh().status = kWalkOverflow;
      } else {
        const int e = walk_sh().nedges++;
        rec->e_dst[e] = walk_sh().ncols;
        rec->e_src[e] = src;
        for (int w = 0; w < 8; ++w) rec->e_lbl[(size_t)e * 8 + w] = shift ? walk_sh().lbl8[w] : 0u;
      }
    }
    const Hot h = hot();
    uint32_t m[KW];
    if (shift) {
      Row::load(walk_sh().lbl, h.W, m);
    } else {
#pragma unroll
      for (int i = 0; i < KW; ++i) m[i] = 0xffffffffu;
      Row::valid(m, h.W);
    }
    if (shift)
      scatter<true>(h, h.col[src], h.col[src + 1], m, warp, nw);
    else
      scatter<false>(h, h.col[src], h.col[src + 1], m, warp, nw);
    __syncthreads();
  }

  __device__ void seed(int c) {
    if (threadIdx.x == 0) {
      const uint32_t s = claim(c);
      row_of(s, c)[g.start_item >> 5] |= 1u << (g.start_item & 31);
      mark(c);
    }
    __syncthreads();
  }

  // ------------------------------------------------------------ the sweep
  // Warp: highest set bit of bm at or below `top`, or -1 (bits may be set and
  // cleared meanwhile).
  __device__ static int warp_highest_dirty(const uint32_t* bm, int top) {
    const int lane = threadIdx.x & 31;
    if (top < 0) return -1;
    for (int wtop = top >> 5; wtop >= 0; wtop -= 32) {
      const int w = wtop - lane;
      uint32_t v = (w >= 0) ? vld(bm + w) : 0u;
      if (w == (top >> 5)) v &= (top & 31) == 31 ? 0xffffffffu : ((2u << (top & 31)) - 1u);
      const unsigned any = __ballot_sync(0xffffffffu, v != 0);
      if (any) {
        const int l = __ffs(any) - 1;
        const uint32_t vv = __shfl_sync(0xffffffffu, v, l);
        return ((wtop - l) << 5) + (31 - __clz(vv));
      }
    }
    return -1;
  }

  // Warp: the nonterminals with a complete item in row (lane v < VW: word v).
  __device__ static __forceinline__ uint32_t completed(const Hot& h, const uint32_t* row) {
    if constexpr (LR == 4) return warp_ntset(row, h.c_off, h.c_lst, h.V, h.VW);
    return warp_completed(row, h.w4, h.m4, h.c_off, h.c_lst, h.V, h.VW);
  }

  // Warp: close row o with its self-loop and scatter the nonterminals that it
  // newly completes over the other entries of column o.
  __device__ static __forceinline__ void visit(const Hot& h, int o, int mode) {
    const int W = h.W, VW = h.VW;
    const int lane = threadIdx.x & 31, li = Row::li();
    const uint32_t s = h.slot(o);
    uint32_t* bd = h.done_of(s, o);
    // done before the row: a visit writes its row before it records what it
    // completed (those were scattered, and advanced in this row, already)
    uint32_t known = (lane < VW) ? vld(bd + lane) : 0u;
    __threadfence_block();
    // every lane group holds a copy of the row
    uint32_t r[KW], r0[KW], e[KW], ex[KW];
    const int kb = h.col[o], ke = h.col[o + 1];
    const bool self = (h.selfb[o >> 5] >> (o & 31)) & 1u;  // the last entry: origins ascend
    const uint32_t s_row = h.s_rows + s * (uint32_t)(W * 4);
    const bool in_smem = s < (uint32_t)h.R;
    if (in_smem) {
      Row::load_shared(s_row, W, r);
    } else {
#pragma unroll
      for (int i = 0; i < KW; ++i) r[i] = li * KW + i < W ? vld(h.stage + (size_t)o * W + li * KW + i) : 0u;
    }
    if (self) {
      Row::load(h.bits + (size_t)(ke - 1) * W, W, e);
    } else {
#pragma unroll
      for (int i = 0; i < KW; ++i) e[i] = 0u;
    }
#pragma unroll
    for (int i = 0; i < KW; ++i) r0[i] = r[i];
    // what the row completes, and everything that follows from it through the
    // self entry, at once (lane v < VW: word v)
    uint32_t tot = 0;
    Row::advance(r, h.adv, mode, h.steps, h.nullable, W);
    uint32_t cm[KW];
    Row::load(h.complete, W, cm);
    bool any = false;
#pragma unroll
    for (int i = 0; i < KW; ++i) {
      cm[i] &= r[i];
      any |= cm[i] != 0;
    }
    if (__any_sync(0xffffffffu, any)) {
      if (lane < LR) Row::store(h.scr, W, cm);
      __syncwarp();
      tot = completed(h, h.scr) & ~known;
      __syncwarp();
      if (__any_sync(0xffffffffu, tot != 0)) {
        const int kind = 2 * (int)((h.gapb[o >> 5] >> (o & 31)) & 1u) + mode;
        tot = warp_follow(tot, h.follow + (size_t)kind * h.V * VW, VW) & ~known;
        Row::waiting_on(tot, h.exp_nt, h.next_t, h.scr, W, VW, ex);
#pragma unroll
        for (int i = 0; i < KW; ++i) e[i] &= ex[i];
        Row::shift_up(e);
#pragma unroll
        for (int i = 0; i < KW; ++i) r[i] |= e[i];
        Row::advance(r, h.adv, mode, h.steps, h.nullable, W);
      }
    }
    if (lane < LR) {
#pragma unroll
      for (int i = 0; i < KW; ++i)
        if (r[i] & ~r0[i]) {
          if (in_smem)
            gs_red_or(s_row + (uint32_t)(li * KW + i) * 4u, r[i]);
          else
            atomicOr(h.stage + (size_t)o * W + li * KW + i, r[i]);
        }
    }
    if (!__any_sync(0xffffffffu, tot != 0)) return;
    __threadfence_block();
    __syncwarp();
    if (lane < VW && tot) atomicOr(bd + lane, tot);
    scatter<true>(h, kb, self ? ke - 1 : ke, ex, 0, 1);
  }

  // Block: close the origins below c (every warp returns when nothing is
  // dirty and no warp holds an origin).
  __device__ void close_origins(int c, int mode) {
    const Hot h = hot();
    const int lane = threadIdx.x & 31;
    const volatile int32_t* busy = &walk_gs().busy;
    long long visits = 0, idle = 0;
    for (;;) {
      // claim the highest dirty origin; a holder counts itself busy before
      // its claim clears the bit, so "no holder, then nothing dirty" means done
      int o = -1;
      for (int tries = 0; tries < 64; ++tries) {
        const int h = warp_highest_dirty(walk_sh().dirty, c - 1);
        if (h < 0) break;
        uint32_t old = 0;
        if (lane == 0) {
          atomicAdd(&walk_gs().busy, 1);
          __threadfence_block();
          old = atomicAnd(&walk_sh().dirty[h >> 5], ~(1u << (h & 31)));
          if (!((old >> (h & 31)) & 1u)) atomicSub(&walk_gs().busy, 1);
        }
        old = __shfl_sync(0xffffffffu, old, 0);
        if ((old >> (h & 31)) & 1u) {
          o = h;
          break;
        }
      }
      if (o < 0) {
        int b = 0;
        if (lane == 0) b = *busy;
        b = __shfl_sync(0xffffffffu, b, 0);
        __threadfence_block();
        if (b == 0 && warp_highest_dirty(walk_sh().dirty, c - 1) < 0) break;
        if (++idle > kGsMaxIdle) {
          if (lane == 0) walk_sh().status = kWalkOverflow;
          break;
        }
        __nanosleep(40);
        continue;
      }
      __syncwarp();  // the claim (lane 0) before any lane reads the row
      __threadfence_block();
      if (++visits <= kGsMaxSteps) {
        visit(h, o, mode);
      } else if (lane == 0) {
        walk_sh().status = kWalkOverflow;
      }
      __threadfence_block();
      __syncwarp();
      if (lane == 0) atomicSub(&walk_gs().busy, 1);
      __syncwarp();
      if (visits > kGsMaxSteps) break;
    }
  }

  // Closure of column c (gap: a node with a Sigma_lex* self-loop).
  __device__ __noinline__ void close_column(int c, bool gap) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = nwarps();
    if (threadIdx.x == 0) {
      if (REC) rec->col_gap[c] = gap ? 1 : 0;
      if (gap) gapb[c >> 5] |= 1u << (c & 31);
    }
    const int mode = gap ? 1 : 0;  // the advance rule: next_any in a gap, nullable_next elsewhere
    // 1. origins below c.  A node (not a gap) reached only by epsilon edges
    //    from finished columns needs no sweep: each of its rows is a union of
    //    rows that are closed under completion and advance, and so is the
    //    union (what an origin completes here, it completed in one of the
    //    sources, whose rows below already hold the advanced items).
    PH_BEGIN(t_or);
    if (gap || walk_gs().labelled) {
      if (threadIdx.x == 0) walk_gs().busy = 0;
      __syncthreads();
      close_origins(c, mode);
    }
    for (int w = threadIdx.x; w < W; w += blockDim.x) walk_gs().uni[w] = 0;
    __syncthreads();
    PH_END(8, t_or);
    if (walk_sh().status == kWalkOverflow) return;
    // 2. predictions: nonterminals waited on by any row of the column
    PH_BEGIN(t_pr);
    bitmap_to_list(walk_sh().touched, c + 1);
    const int nl = walk_sh().list_n;
    {
      uint32_t acc[KW];
#pragma unroll
      for (int i = 0; i < KW; ++i) acc[i] = 0u;
      for (int i = warp * NG + Row::gi(); i < nl; i += nw * NG) {
        const int o = walk_sh().list[i];
        uint32_t v[KW];
        Row::load(row_of(slot(o), o), W, v);
#pragma unroll
        for (int j = 0; j < KW; ++j) acc[j] |= v[j];
      }
      uint32_t an[KW];
      Row::load(tb.any_nt, W, an);
#pragma unroll
      for (int j = 0; j < KW; ++j)
        if (acc[j] & an[j]) atomicOr(&walk_gs().uni[Row::li() * KW + j], acc[j] & an[j]);
    }
    __syncthreads();
    const int32_t* w_off = plan.o_wait ? (const int32_t*)(gs_smem() + plan.o_woff) : g.wait_off;
    const uint2* w_lst = plan.o_wait ? (const uint2*)(gs_smem() + plan.o_wait) : g.wait;
    for (int v = warp; v < VW; v += nw) {  // one warp per word of the set
      const int A = (v << 5) + lane;
      bool hit = false;
      if (A < g.V)
        for (int q = w_off[A], e = w_off[A + 1]; q < e && !hit; ++q) {
          const uint2 p = w_lst[q];
          hit = (walk_gs().uni[p.x] & p.y) != 0;
        }
      const uint32_t b = __ballot_sync(0xffffffffu, hit);
      if (lane == 0) walk_gs().vset[v] = b;
    }
    if (threadIdx.x == 0) claim(c);
    __syncthreads();
    uint32_t* crow = row_of(slot(c), c);
    {
      const uint32_t* P = gap ? g.gap_pred : g.pred;
      uint32_t acc[KW];
#pragma unroll
      for (int i = 0; i < KW; ++i) acc[i] = 0u;
      // the warps' lane groups share out the nonterminals
      const int part = warp * NG + Row::gi(), parts = nw * NG;
      int seen = 0;
      for (int v = 0; v < VW; ++v) {
        uint32_t m = walk_gs().vset[v];
        while (m) {
          const int b0 = __ffs(m) - 1;
          m &= m - 1;
          if (seen++ % parts != part) continue;
          uint32_t x[KW];
          Row::load(P + (size_t)((v << 5) + b0) * W, W, x);
#pragma unroll
          for (int i = 0; i < KW; ++i) acc[i] |= x[i];
        }
      }
      bool nz = false;
#pragma unroll
      for (int i = 0; i < KW; ++i)
        if (acc[i]) {
          atomicOr(crow + Row::li() * KW + i, acc[i]);
          nz = true;
        }
      if (__any_sync(0xffffffffu, nz) && lane == 0) atomicOr(&walk_sh().touched[c >> 5], 1u << (c & 31));
    }
    __syncthreads();
    // a seeded row c (the walk's first column) is closed by the advance rule
    if (warp == 0 && bit_get(walk_sh().dirty, c)) {
      uint32_t r[KW];
      Row::load(crow, W, r);
      Row::advance(r, tb.adv_pow, mode, g.adv_steps, g.any_nullable, W);
      __syncwarp();
      if (lane < LR) Row::store(crow, W, r);
    }
    __syncthreads();
    PH_END(10, t_pr);
  }

  // Move the rows of the open column into the entry store as column c
  // (origins ascending), recording completed nonterminals.  A touched row is
  // never empty.
  __device__ __noinline__ void finish_column(int c) {
    PH_BEGIN(t_fi);
    const int warp = threadIdx.x >> 5, nw = nwarps();
    bitmap_to_list(walk_sh().touched, c + 1);
    const int nl = walk_sh().list_n;
    const int base = ws.col_off[c];
    const bool ok = (long long)base + nl <= dims.emax;
    if (threadIdx.x == 0) {
      if (!ok) {
        walk_sh().status = kWalkOverflow;
      } else {
        ws.col_off[c + 1] = base + nl;
        walk_sh().nent = base + nl;
      }
      walk_sh().ncols = c + 1;
      walk_gs().labelled = 0;
      walk_gs().nslots = 0;
    }
    if constexpr (REC) {
      const Hot h = hot();
      if (ok)
        for (int i = warp; i < nl; i += nw) {
          const int o = walk_sh().list[i];
          record_entry(h, row_of(slot(o), o), (size_t)base + i);
        }
    }
    if (REC) __syncthreads();  // rows are cleared below, by other warps than read them here
    // one lane group per row
    for (int i = warp * NG + Row::gi(); i < nl; i += nw * NG) {
      const int o = walk_sh().list[i];
      const uint32_t s = slot(o);
      uint32_t* row = row_of(s, o);
      uint32_t v[KW];
      Row::load(row, W, v);
      if (ok) {
        const size_t k = (size_t)base + i;
        Row::store(ws.bits + k * W, W, v);
        if (Row::li() == 0) {
          ws.org[k] = o;
          if (o == c) selfb[c >> 5] |= 1u << (c & 31);  // one group holds origin c
        }
      }
#pragma unroll
      for (int j = 0; j < KW; ++j) v[j] = 0u;
      Row::store(row, W, v);
      uint32_t* bd = done_of(s, o);
      for (int w = Row::li(); w < VW; w += LR) bd[w] = 0;
      if (Row::li() == 0) slot_of[o] = (uint16_t)kSlotNone;
    }
    __syncthreads();
    if (threadIdx.x == 0) slot_of[c] = (uint16_t)kSlotNone;  // claimed even if nothing was predicted
    clear_bitmap(walk_sh().touched, c + 1);
    clear_bitmap(walk_sh().dirty, c + 1);
    __syncthreads();
    PH_END(11, t_fi);
  }

  __device__ bool column_empty(int c) const { return ws.col_off[c + 1] == ws.col_off[c]; }

  // Warp: completed nonterminals of entry k, its row in memory.
  __device__ __forceinline__ void record_entry(const Hot& h, const uint32_t* row, size_t k) {
    const int lane = threadIdx.x & 31;
    const uint32_t cn = completed(h, row);
    if (lane < VW) rec->cnt[k * VW + lane] = cn;
  }

  // After an aborted walk: return the rows of the open column to zero.
  __device__ void cleanup() {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = nwarps();
    __syncthreads();
    for (int o = warp; o < dims.nmax; o += nw) {
      const uint32_t s = slot(o);
      if (s == kSlotNone) continue;
      uint32_t* row = row_of(s, o);
      for (int w = lane; w < W; w += 32) row[w] = 0;
      uint32_t* bd = done_of(s, o);
      for (int v = lane; v < VW; v += 32) bd[v] = 0;
      __syncwarp();
      if (lane == 0) slot_of[o] = (uint16_t)kSlotNone;
    }
    if (threadIdx.x == 0) {
      walk_gs().labelled = 0;
      walk_gs().nslots = 0;
    }
    clear_bitmap(walk_sh().touched, kMaxCols);
    clear_bitmap(walk_sh().dirty, kMaxCols);
    __syncthreads();
  }

  __device__ bool accepts(int c, int start_col) {
    __shared__ int found;
    if (threadIdx.x == 0) found = 0;
    __syncthreads();
    for (int k = ws.col_off[c] + threadIdx.x; k < ws.col_off[c + 1]; k += blockDim.x)
      if (ws.org[k] == start_col && bit_get(ws.bits + (size_t)k * W, g.accept_item)) found = 1;
    __syncthreads();
    return found != 0;
  }
};

}  // namespace epic
