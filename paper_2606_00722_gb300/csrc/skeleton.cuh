// The graph walk shared by exact recognition (EarleyColsGS) and the cover
// group test (CoverCols): it enumerates the nodes of the partial-output graph
// of x (+) Delta in topological order, building them from the lex table, and
// asks the column type to combine, close and store each node.
#pragma once
#include "cover.cuh"
#include "walk.cuh"

namespace epic {

template <class Cols>
struct Walk {
  Cols& cols;
  const DevGrammar& g;
  const LexEntry* table;
  WalkScratch sc;
  int vocab;
  const BlockRec* rec = nullptr;  // recording walks: positions' columns

  __device__ Walk(Cols& c, const DevGrammar& g_, const LexEntry* t, WalkScratch s, int v)
      : cols(c), g(g_), table(t), sc(s), vocab(v) {}

  __device__ __noinline__ void label_set(const uint32_t* lbl8) {
    if (Cols::kRecord && threadIdx.x < 8) walk_sh().lbl8[threadIdx.x] = lbl8[threadIdx.x];
    for (int w = threadIdx.x; w < g.W; w += blockDim.x) walk_sh().lbl[w] = 0;
    __syncthreads();
    // the terminals are shared out among the warps
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    uint32_t share = 0;
    for (int b = warp; b < 32; b += nw) share |= 1u << b;
    for (int lw = 0; lw < 8; ++lw) {
      uint32_t m = lbl8[lw] & share;
      while (m) {
        const int a = (lw << 5) + __ffs(m) - 1;
        m &= m - 1;
        if (a >= g.T) continue;
        for (int w = lane; w < g.W; w += 32) {
          const uint32_t v = g.exp_term[(size_t)a * g.W + w];
          if (v) atomicOr(&walk_sh().lbl[w], v);
        }
      }
    }
    __syncthreads();
  }
  __device__ void label_one(int a) {
    if (Cols::kRecord && threadIdx.x < 8) walk_sh().lbl8[threadIdx.x] = (threadIdx.x == (a >> 5)) ? (1u << (a & 31)) : 0u;
    for (int w = threadIdx.x; w < g.W; w += blockDim.x) walk_sh().lbl[w] = g.exp_term[(size_t)a * g.W + w];
    __syncthreads();
  }

  __device__ static int token_at(const int32_t* x, const Subst& s, int i) {
    for (int j = 0; j < s.n; ++j)
      if (s.pos[j] == i) return s.tok[j];
    return x[i];
  }

  // Arrival of group gi into its end node: (source column, label set), the
  // label set all zero for an epsilon edge.
  __device__ int arrival_src(int gi) const { return sc.g_len[gi] >= 2 ? sc.g_last[gi] : sc.g_src[gi]; }
  __device__ uint32_t arrival_lbl(int gi, int w) const {
    const int len = sc.g_len[gi];
    if (len == 0) return 0u;
    if (len == 1) return sc.g_lbl[gi * 8 + w];
    const int a = sc.g_tail[gi * 16 + len - 2];
    return (w == (a >> 5)) ? (1u << (a & 31)) : 0u;
  }
  // Do end states e1 and e2 receive the same arrivals?  (One thread.)
  __device__ bool same_arrivals(int e1, int e2, int ng) const {
    int n1 = 0, n2 = 0;
    for (int gi = 0; gi < ng; ++gi) {
      n1 += sc.g_end[gi] == e1;
      n2 += sc.g_end[gi] == e2;
    }
    if (n1 != n2) return false;
    for (int gi = 0; gi < ng; ++gi) {
      if (sc.g_end[gi] != e1) continue;
      bool found = false;
      for (int gj = 0; gj < ng && !found; ++gj) {
        if (sc.g_end[gj] != e2 || arrival_src(gj) != arrival_src(gi)) continue;
        bool same = (sc.g_len[gi] == 0) == (sc.g_len[gj] == 0);
        for (int w = 0; w < 8; ++w) same &= arrival_lbl(gi, w) == arrival_lbl(gj, w);
        found = same;
      }
      if (!found) return false;
    }
    return true;
  }

  // Block: index of element i's bit among the set bits of walk_sh().qbits.
  __device__ int rank_of(int i) const {
    int r = __popc(walk_sh().qbits[i >> 5] & ((1u << (i & 31)) - 1u));
    for (int w = 0; w < (i >> 5); ++w) r += __popc(walk_sh().qbits[w]);
    return r;
  }
  __device__ int count_set(int nbits) const {
    int r = 0;
    for (int w = 0; w < ((nbits + 31) >> 5); ++w) r += __popc(walk_sh().qbits[w]);
    return r;
  }
  // the first terminal does not separate lexings (bits 24..31 of the word)
  __device__ static bool same_lexing(const uint4& a, const uint4& b) {
    return ((a.x ^ b.x) & 0x00FFFFFFu) == 0 && a.y == b.y && a.z == b.z && a.w == b.w;
  }

  // One token of a span: frontier (f_q lexer state, f_c column)[0..nf) ->
  // new frontier.  Lexings from the same column with the same end state and
  // the same terminals after the first share one path whose first edge
  // carries all their first terminals.  Every step but the columns
  // themselves is one thread per lexing, group or end state over the shared
  // tables (after a gap the frontier is every lexer state, and one thread
  // walking such lists took longer than the columns).  Returns false on
  // overflow.
  __device__ __noinline__ bool span_step(int tok) {
    const int nf = walk_sh().nf, nthr = blockDim.x, tid = threadIdx.x;
    const WalkScratch sc = this->sc;  // in registers across the barriers
    if (g.lazy.stats && tid == 0) atomicAdd(&g.lazy.stats[0], (unsigned long long)nf);
    for (int f = tid; f < nf; f += nthr) sc.ent[f] = lex_at(g, table, tok, sc.f_q[f]);
    clear_bitmap(walk_sh().qbits, kMaxQ);
    __syncthreads();
    // each live lexing's leader: the first one with its key
    const uint4* ent = (const uint4*)sc.ent;
    for (int f = tid; f < nf; f += nthr) {
      int leader = -1;
      if (sc.ent[f].end != 0xFFFF) {
        const uint4 e = ent[f];
        const int src = sc.f_c[f];
        leader = 0;
        while (leader < f && !(sc.f_c[leader] == src && same_lexing(ent[leader], e))) ++leader;
        if (leader == f) atomicOr(&walk_sh().qbits[f >> 5], 1u << (f & 31));
      }
      sc.key_q[f] = leader;
    }
    __syncthreads();
    const int ng = count_set(nf);
    for (int f = tid; f < nf; f += nthr) {
      if (sc.key_q[f] != f) continue;
      const int gi = rank_of(f);
      const LexEntry e = sc.ent[f];
      sc.g_src[gi] = sc.f_c[f];
      sc.g_end[gi] = e.end;
      sc.g_len[gi] = e.len;
      for (int t = 0; t < 16; ++t) sc.g_tail[gi * 16 + t] = (t + 1 < e.len) ? e.term[t + 1] : 0;
      for (int w = 0; w < 8; ++w) sc.g_lbl[gi * 8 + w] = 0;
    }
    __syncthreads();
    for (int f = tid; f < nf; f += nthr) {
      const int k = sc.key_q[f];
      if (k < 0 || sc.ent[f].len == 0) continue;
      const int a = sc.ent[f].term[0];
      atomicOr(&sc.g_lbl[rank_of(k) * 8 + (a >> 5)], 1u << (a & 31));
    }
    __syncthreads();
    // the run up to its last terminal (intermediate nodes); groups with the
    // same source, first-terminal set and terminals before the last one
    // spell the same paths up to it, so they share one chain of nodes (key_q:
    // the group whose chain this one takes, -1: its own)
    for (int gi = tid; gi < ng; gi += nthr) {
      const int len = sc.g_len[gi], src = sc.g_src[gi];
      int share = -1;
      if (len >= 2)
        for (int gj = 0; gj < gi && share < 0; ++gj) {
          if (sc.g_len[gj] != len || sc.g_src[gj] != src) continue;
          bool same = true;
          for (int w = 0; w < 8; ++w) same &= sc.g_lbl[gj * 8 + w] == sc.g_lbl[gi * 8 + w];
          for (int t = 0; t + 2 < len; ++t) same &= sc.g_tail[gj * 16 + t] == sc.g_tail[gi * 16 + t];
          if (same) share = gj;
        }
      sc.key_q[gi] = share;
    }
    __syncthreads();
    for (int gi = 0; gi < ng; ++gi) {
      const int len = sc.g_len[gi];
      int cur = sc.g_src[gi];
      if (sc.key_q[gi] >= 0) continue;
      for (int t = 0; t + 1 < len; ++t) {
        int c = cols.open_column();
        __syncthreads();
        if (c < 0) return false;
        if (t == 0)
          label_set(sc.g_lbl + gi * 8);
        else
          label_one(sc.g_tail[gi * 16 + t - 1]);
        cols.arrive_labels(cur, false);
        cols.close_column(c, false);
        cols.finish_column(c);
        if (walk_sh().status != kWalkOk) return false;
        cur = c;
      }
      if (tid == 0) sc.g_last[gi] = cur;
    }
    clear_bitmap(walk_sh().qbits, kMaxQ);
    __syncthreads();
    for (int gi = tid; gi < ng; gi += nthr) {
      if (sc.key_q[gi] >= 0) sc.g_last[gi] = sc.g_last[sc.key_q[gi]];  // chains have owners, not chains of chains
      atomicOr(&walk_sh().qbits[sc.g_end[gi] >> 5], 1u << (sc.g_end[gi] & 31));
    }
    __syncthreads();
    // one node per distinct end state, ascending
    const int nt = count_set(g.Q);
    for (int q = tid; q < g.Q; q += nthr)
      if ((walk_sh().qbits[q >> 5] >> (q & 31)) & 1u) sc.f_q[rank_of(q)] = q;
    __syncthreads();
    // end nodes with the same arrivals (sources and labels) have the same
    // incoming paths: one column serves all their lexer states.  Each end's
    // arrivals are hashed and counted; the smallest equal end is its
    // representative (key_q).
    for (int ti = tid; ti < nt; ti += nthr) {
      const int e = sc.f_q[ti];
      uint32_t h = 0;
      int cnt = 0;
      for (int gi = 0; gi < ng; ++gi) {
        if (sc.g_end[gi] != e) continue;
        uint32_t x = (uint32_t)arrival_src(gi) * 0x9E3779B1u + (sc.g_len[gi] == 0 ? 0x85EBCA6Bu : 0u);
        for (int w = 0; w < 8; ++w) x = (x ^ arrival_lbl(gi, w)) * 0xC2B2AE35u + (uint32_t)w;
        h += x ^ (x >> 16);
        ++cnt;
      }
      walk_sh().hash[ti] = h;
      walk_sh().narr[ti] = cnt;
    }
    __syncthreads();
    for (int ti = tid; ti < nt; ti += nthr) {
      int rep = ti;
      for (int tj = 0; tj < ti; ++tj)
        if (walk_sh().hash[tj] == walk_sh().hash[ti] && walk_sh().narr[tj] == walk_sh().narr[ti] && same_arrivals(sc.f_q[ti], sc.f_q[tj], ng)) {
          rep = tj;
          break;
        }
      sc.key_q[ti] = rep;
    }
    __syncthreads();
    for (int ti = 0; ti < nt; ++ti) {
      if (sc.key_q[ti] != ti) continue;
      int e = sc.f_q[ti];
      int c = cols.open_column();
      __syncthreads();
      if (c < 0) return false;
      for (int gi = 0; gi < ng; ++gi) {
        if (sc.g_end[gi] != e) continue;
        int len = sc.g_len[gi];
        if (len == 0) {
          cols.arrive_labels(sc.g_src[gi], true);
        } else if (len == 1) {
          label_set(sc.g_lbl + gi * 8);
          cols.arrive_labels(sc.g_src[gi], false);
        } else {
          label_one(sc.g_tail[gi * 16 + len - 2]);
          cols.arrive_labels(sc.g_last[gi], false);
        }
      }
      cols.close_column(c, false);
      cols.finish_column(c);
      if (walk_sh().status != kWalkOk) return false;
      if (tid == 0) sc.f_c[ti] = c;
      __syncthreads();
    }
    // the new frontier: (end state, column) of the non-empty columns, in order
    if (tid < 32) {
      int k = 0;
      for (int t0 = 0; t0 < nt; t0 += 32) {
        const int ti = t0 + tid;
        int q = 0, c = -1;
        if (ti < nt) {
          q = sc.f_q[ti];
          // a representative is never after its members, and holds its own
          // column until its chunk is compacted
          c = sc.f_c[sc.key_q[ti]];
        }
        const bool live = ti < nt && !cols.column_empty(c);
        const unsigned m = __ballot_sync(0xffffffffu, live);
        if (live) {
          const int at = k + __popc(m & ((1u << tid) - 1u));
          sc.g_src[at] = q;  // the groups are done with
          sc.g_end[at] = c;
        }
        k += __popc(m);
      }
      __syncwarp();
      for (int i = tid; i < k; i += 32) {
        sc.f_q[i] = sc.g_src[i];
        sc.f_c[i] = sc.g_end[i];
      }
      if (tid == 0) walk_sh().nf = k;
    }
    __syncthreads();
    return true;
  }

  // Arrivals of the frontier into the open column: by an epsilon edge, by the
  // pending lexeme's terminal, or none (a dead end); frontier elements with
  // the same column and the same edge arrive once.  At a gap, a pending
  // lexeme that some byte can extend stays open (the gap absorbs its
  // terminal); one that no byte can extend has ended and emits its terminal.
  __device__ __noinline__ void arrive_frontier(bool gap) {
    const int nf = walk_sh().nf;
    for (int f = threadIdx.x; f < nf; f += blockDim.x) {
      const int q = sc.f_q[f], a = g.dfa_accept[q];
      int kind = -2;
      if (q == 0 || (gap && g.dfa_ext[q]) || (a >= 0 && g.skip[a]))
        kind = -1;
      else if (a >= 0)
        kind = a;
      sc.g_len[f] = kind;
    }
    __syncthreads();
    for (int f = threadIdx.x; f < nf; f += blockDim.x) {
      const int kind = sc.g_len[f], c = sc.f_c[f];
      bool dup = false;
      for (int h = 0; h < f && !dup; ++h) dup = sc.f_c[h] == c && sc.g_len[h] == kind;
      sc.key_q[f] = dup ? -2 : kind;
    }
    __syncthreads();
    for (int f = 0; f < nf; ++f) {
      const int kind = sc.key_q[f];
      if (kind == -1) {
        cols.arrive_labels(sc.f_c[f], true);
      } else if (kind >= 0) {
        label_one(kind);
        cols.arrive_labels(sc.f_c[f], false);
      }
    }
  }

  // Walk x (+) s.  Returns 1 (accept item at the accept node), 0, -1 on a
  // capacity overflow, -2 on bad input (unmasked position, bad token id).
  __device__ __noinline__ int run(const int32_t* x, int n, Subst s) {
    cols.reset();
    if (threadIdx.x == 0) {
      for (int j = 0; j < s.n; ++j) {
        int p = s.pos[j];
        if (p < 0 || p >= n || x[p] >= 0 || s.tok[j] < 0 || s.tok[j] >= vocab) walk_sh().status = kWalkBadInput;
      }
    }
    __syncthreads();
    if (walk_sh().status != kWalkOk) return -2;
    int r = run_inner(x, n, s);
    if (r < 0) cols.cleanup();
    return r;
  }

  __device__ int seed_column(bool gap) {
    int c = cols.open_column();
    __syncthreads();
    if (c < 0) return -1;
    if (threadIdx.x == 0) walk_sh().start_col = c;
    __syncthreads();
    cols.seed(c);
    return c;
  }

  // positions [lo, hi) of a recording walk -> column c
  __device__ void rec_range(int32_t* arr, int lo, int hi, int c) {
    for (int p = lo + threadIdx.x; p < hi; p += blockDim.x) arr[p] = c;
  }

  __device__ int run_inner(const int32_t* x, int n, Subst s) {
    if (n == 0) {
      int c = seed_column(false);
      if (c < 0) return -1;
      cols.close_column(c, false);
      cols.finish_column(c);
      if (walk_sh().status != kWalkOk) return -1;
      if (threadIdx.x == 0) walk_sh().accept_col = c;
      return cols.column_has_accept(c, c) ? 1 : 0;
    }
    int i = 0;
    bool first = true;
    int prev_gap = -1;
    int span_lo = -1, span_hi = -1;  // the last span (recording walks)
    while (i < n) {
      int t0 = token_at(x, s, i);
      int j = i;
      if (t0 < 0) {
        while (j < n && token_at(x, s, j) < 0) ++j;
        int c;
        if (first) {
          c = seed_column(true);
          if (c < 0) return -1;
        } else {
          c = cols.open_column();
          __syncthreads();
          if (c < 0) return -1;
          arrive_frontier(true);
        }
        cols.close_column(c, true);
        cols.finish_column(c);
        if (walk_sh().status != kWalkOk) return -1;
        if (Cols::kRecord) {
          rec_range(rec->gap_col, i, j, c);
          if (span_lo >= 0) rec_range(rec->post_col, span_lo, span_hi, c);
        }
        prev_gap = c;
        if (cols.column_empty(c)) return 0;
      } else {
        while (j < n && token_at(x, s, j) >= 0) ++j;
        if (first) {
          int c = seed_column(false);
          if (c < 0) return -1;
          cols.close_column(c, false);
          cols.finish_column(c);
          if (walk_sh().status != kWalkOk) return -1;
          if (threadIdx.x == 0) {
            sc.f_q[0] = 0;
            sc.f_c[0] = c;
            walk_sh().nf = 1;
          }
          if (Cols::kRecord) rec_range(rec->pre_col, i, j, c);
        } else {
          if (Cols::kRecord) rec_range(rec->pre_col, i, j, prev_gap);
          for (int q = threadIdx.x; q < g.Q; q += blockDim.x) {
            sc.f_q[q] = q;
            sc.f_c[q] = prev_gap;
          }
          if (threadIdx.x == 0) walk_sh().nf = g.Q;
        }
        __syncthreads();
        span_lo = i;
        span_hi = j;
        for (int p = i; p < j; ++p) {
          if (walk_sh().nf == 0) break;
          int tok = token_at(x, s, p);
          if (tok < 0 || tok >= vocab) return -2;
          if (!span_step(tok)) return -1;
        }
        if (walk_sh().nf == 0) return 0;  // no lexing of this span survives
        if (j == n) {              // END: flush the pending lexeme
          int c = cols.open_column();
          __syncthreads();
          if (c < 0) return -1;
          arrive_frontier(false);
          cols.close_column(c, false);
          cols.finish_column(c);
          if (walk_sh().status != kWalkOk) return -1;
          if (Cols::kRecord) rec_range(rec->post_col, i, j, c);
          if (threadIdx.x == 0) walk_sh().accept_col = c;
          return cols.column_has_accept(c, walk_sh().start_col) ? 1 : 0;
        }
      }
      first = false;
      i = j;
    }
    if (threadIdx.x == 0) walk_sh().accept_col = prev_gap;
    return cols.column_has_accept(prev_gap, walk_sh().start_col) ? 1 : 0;
  }
};

}  // namespace epic
