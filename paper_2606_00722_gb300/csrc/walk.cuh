// Block-wide Earley recognition over the lexeme graph of a partial output
// (Alg. 3 on the graph of Alg. 2), built on the fly from the lex table.
//
// The graph (the gap reading): every maximal run of masks is a gap node with a
// self-loop on every terminal; every maximal run of tokens is a span whose
// lexings are paths.  Inside a span the graph nodes are (token boundary,
// lexer state) pairs -- lexings that reach the same lexer state at the same
// token boundary continue identically, so they share the node -- plus one
// node per distinct (target, remaining run) between boundaries, so that runs
// that differ only in their first terminal share the rest of their path.
// The paths between two nodes spell exactly the distinct terminal runs of the
// span from its entry states (q0 at the sequence start, every lexer state
// after a gap), flushed at END; so the language of the graph, and hence the
// validity bit, is that of the per-alternative graph of the definition.
//
// Chart (Alg. 3 items): for every graph node c, a list of entries (origin
// node o, bitset over dotted items) -- the items (p, d, o) present at c.
// Predict / scan / complete are bit-parallel: a scan over terminal a is
// ((bits & EXP_T[a]) << 1) because item (p, d+1) follows item (p, d); a
// completion of the nonterminals Bset from origin o' advances the items
// of column o' that wait on a member of Bset; prediction ORs precomputed
// prediction closures; nullable nonterminals are skipped on prediction
// (Aycock & Horspool); inside a gap every item advances over any symbol.
#pragma once
#include "device.cuh"

namespace epic {

constexpr int kMaxCols = 4096;   // columns (graph nodes) per walk
constexpr int kMaxQ = 1024;      // lexer states
constexpr int kMaxW = 256;       // item words (D <= 8192)
constexpr int kMaxVW = 32;       // nonterminal words (V <= 1024)

enum WalkStatus { kWalkOk = 0, kWalkOverflow = 1, kWalkBadInput = 2, kWalkDead = 3 };

struct Subst {   // (position, token) substitutions, sorted by position
  const int32_t* pos;
  const int32_t* tok;
  int n;
};

// Per-walk tables of the span step (shared memory when the lexer is small
// enough, else the global workspace): the groups of lexings of one token and
// the frontier.
struct WalkScratch {
  int32_t* g_src;     // [kMaxQ] group source column
  int32_t* g_end;     // [kMaxQ] group end lexer state
  int32_t* g_len;     // [kMaxQ]
  uint8_t* g_tail;    // [kMaxQ][16] terminals after the first
  uint32_t* g_lbl;    // [kMaxQ][8] first-terminal label set
  int32_t* g_last;    // [kMaxQ] column holding the run before its last terminal
  int32_t* f_q;       // [kMaxQ] frontier lexer states
  int32_t* f_c;       // [kMaxQ] frontier columns
  int32_t* key_q;     // [kMaxQ] leader of a lexing, shared chain of a group, representative of an end node
  LexEntry* ent;      // [kMaxQ] the token's lex entries from the frontier's states
};

struct WalkShared {
  uint32_t touched[kMaxCols / 32];
  uint32_t dirty[kMaxCols / 32];
  uint16_t list[kMaxCols];
  int32_t before[kMaxCols / 32];
  int32_t list_n;
  uint32_t hash[kMaxQ];       // span step: arrivals of each end node, hashed ...
  int32_t narr[kMaxQ];        // ... and counted
  uint32_t qbits[kMaxQ / 32]; // span step: set over frontier elements or lexer states
  alignas(16) uint32_t lbl[kMaxW];
  int32_t ncols;
  long long nent;
  int32_t status;
  int32_t nf;
  int32_t start_col, accept_col;
  int32_t nedges;    // edges recorded so far (recording walks)
  uint32_t lbl8[8];  // terminal set of the arrivals being made
  int32_t scratch_i[4];
};

// The CTA walks' shared state lies at the start of the kernels' dynamic shared
// memory: a fixed address, so that code inside calls reaches it with plain
// shared-memory instructions and no pointer to reload after each barrier.
struct GsShared {
  uint32_t vset[kMaxVW];             // nonterminals waited on in this column
  alignas(16) uint32_t uni[kMaxW];   // union of the column's rows (items waiting on nonterminals)
  int32_t labelled;                  // the open column has a labelled arrival (else only epsilon ones)
  int32_t busy;                      // warps holding an origin
  int32_t nslots;                    // row slots handed out in the open column
};
struct WalkSmem {
  WalkShared sh;
  GsShared gs;
};
constexpr uint32_t kWalkSmemBytes = (uint32_t)((sizeof(WalkSmem) + 15) & ~(size_t)15);
// the kernels' dynamic shared memory (a name, so that accesses compile to
// shared-memory instructions also inside calls)
__device__ __forceinline__ unsigned char* gs_smem() {
  extern __shared__ __align__(16) unsigned char dyn[];
  return dyn;
}
__device__ __forceinline__ WalkShared& walk_sh() { return reinterpret_cast<WalkSmem*>(gs_smem())->sh; }
__device__ __forceinline__ GsShared& walk_gs() { return reinterpret_cast<WalkSmem*>(gs_smem())->gs; }

__device__ __forceinline__ bool bit_get(const uint32_t* m, int i) { return (m[i >> 5] >> (i & 31)) & 1u; }

// ------------------------------------------------------------ block helpers
// Compact the set bits of bitmap[0 .. nbits) into sh.list (ascending).
__device__ inline void bitmap_to_list(const uint32_t* bitmap, int nbits) {
  WalkShared& sh = walk_sh();
  const int nw = (nbits + 31) >> 5;
  if (threadIdx.x < 32) {  // bits before each word
    const int lane = threadIdx.x;
    int base = 0;
    for (int w0 = 0; w0 < nw; w0 += 32) {
      const int c = w0 + lane < nw ? __popc(bitmap[w0 + lane]) : 0;
      int s = c;
      for (int off = 1; off < 32; off <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, s, off);
        if (lane >= off) s += t;
      }
      if (w0 + lane < nw) sh.before[w0 + lane] = base + s - c;
      base += __shfl_sync(0xffffffffu, s, 31);
    }
    if (lane == 0) sh.list_n = base;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nw * 32; i += blockDim.x) {
    const uint32_t m = bitmap[i >> 5];
    if ((m >> (i & 31)) & 1u) sh.list[sh.before[i >> 5] + __popc(m & ((1u << (i & 31)) - 1u))] = (uint16_t)i;
  }
  __syncthreads();
}

__device__ __forceinline__ void clear_bitmap(uint32_t* bm, int nbits) {
  for (int w = threadIdx.x; w < ((nbits + 31) >> 5); w += blockDim.x) bm[w] = 0;
}

// What a recording walk (a sequence's forward chart, for checks by region)
// writes besides the chart: the graph's edges in target order with their
// terminal sets (all zero: epsilon), gap flags, each entry's completed
// nonterminals, and the column before, at and after each position's segment.
struct BlockRec {
  uint8_t* col_gap;   // [nmax]
  int32_t* e_dst;     // [edge_cap]
  int32_t* e_src;     // [edge_cap]
  uint32_t* e_lbl;    // [edge_cap][8]
  uint32_t* cnt;      // [emax][VW]
  int32_t* gap_col;   // [n]
  int32_t* pre_col;   // [n]
  int32_t* post_col;  // [n]
  int edge_cap;
};

}  // namespace epic
