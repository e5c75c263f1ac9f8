// Kernels and C-ABI of the EPIC hot path on sm_103a (see include/epic.h).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <mutex>
#include <new>
#include <stdexcept>
#include <string>
#include <vector>

#include "../../include/epic.h"
#include "../../include/epic_measure.h"
#include "grammar.h"
#include "launch.h"

using namespace epic;

// ================================================================ kernels

// K1: memoized lex table.  One thread per (token, entry state); consecutive
// threads share a token (its bytes are a broadcast read) and write
// consecutive 16-byte entries.
__global__ void k_lex_table(const int32_t* __restrict__ tok_off, const uint8_t* __restrict__ bytes, int vocab,
                            int Q, const int32_t* __restrict__ dfa_next, const int16_t* __restrict__ dfa_acc,
                            const uint8_t* __restrict__ skip, LexEntry* __restrict__ table, int* overflow) {
  long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)vocab * Q) return;
  int t = (int)(idx / Q), q = (int)(idx % Q);
  bool ovf = false;
  const LexEntry e = lex_transduce(bytes, tok_off[t], tok_off[t + 1], q, dfa_next, dfa_acc, skip, &ovf);
  if (ovf) atomicExch(overflow, 1);
  table[idx] = e;
}

// Per proposed position: the highest-confidence candidate with valid bit 1.
__global__ void k_pick(const int32_t* __restrict__ cand, const float* __restrict__ conf,
                       const uint8_t* __restrict__ valid, int B, int k, int K, int32_t* __restrict__ tok,
                       float* __restrict__ out_conf) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)B * k) return;
  int best = -1;
  float bc = 0.f;
  for (int c = 0; c < K; ++c) {
    long long q = i * K + c;
    if (valid[q] != 1) continue;
    float v = conf[q];
    if (best < 0 || v > bc) {
      best = c;
      bc = v;
    }
  }
  tok[i] = best < 0 ? -1 : cand[i * K + best];
  out_conf[i] = best < 0 ? 0.f : bc;
}

__global__ void k_commit(int32_t* __restrict__ x, int B, int n, const int32_t* __restrict__ pos, int k,
                         const int32_t* __restrict__ tok, const uint8_t* __restrict__ sel) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)B * k) return;
  if (sel[i] != 1) return;
  long long b = i / k;
  int p = pos[i];
  if (p >= 0 && p < n) x[b * n + p] = tok[i];
}

// ================================================================ host side

struct epic_grammar {
  int device = 0;
  GrammarTables tabs;
  LexerDFA dfa;
  CoverTables cov;
  DevGrammar dg{};
  std::vector<void*> dev_allocs;
};

struct epic_lexer_table {
  const epic_grammar* g = nullptr;
  int vocab = 0;
  LexEntry* d_table = nullptr;  // dense tables; null for lazy ones
  // the grammar's device tables with this table's lazy memo (keys null: dense)
  DevGrammar dgl{};
  uint32_t* d_lz_keys = nullptr;  // lazy memo (Alg. 2's cache filled on use)
  uint32_t* d_lz_ready = nullptr;
  LexEntry* d_lz_vals = nullptr;
  int32_t* d_lz_off = nullptr;
  uint8_t* d_lz_bytes = nullptr;
  long long lz_cap = 0;
  char* d_ws = nullptr;
  size_t ws_bytes = 0;
  WsDims dims{};
  int ctas = 0;
  unsigned long long* d_stats = nullptr;
  mutable unsigned long long n_region = 0, n_vkernels = 0;  // host-side counters
  unsigned long long* d_counter = nullptr;
  int8_t* d_spec = nullptr;  // speculative Alg. 4 answers, 2 per sequence
  char* d_seq = nullptr;     // per-sequence forward charts (region checks)
  size_t seq_bytes = 0;
  int32_t* d_regs = nullptr; // per-warp tables of region checks
  char* d_wit = nullptr;     // witness extraction: goals and stack per sequence
  size_t wit_bytes = 0;
  char* d_fb = nullptr;      // rejection fallback: rejections, state and round results per sequence
  size_t fb_bytes = 0;
  mutable unsigned long long n_fb_rounds = 0;  // host-side counter: fallback rounds launched
  size_t regs_bytes = 0;
  int spec_cap = 0;
  char* d_wws = nullptr;   // warp-walk workspace
  size_t wws_bytes = 0;
  int wnmax = 0;
  long long wemax = 0;
  int wwarps = 0;
  cudaStream_t last = nullptr;
  // workspaces that launches under stream capture were given: a graph may
  // replay them, so they are kept until the table goes, also when replaced
  std::vector<void*> in_graphs;
  // CUDA events around the kernels of the last epic_validate_batch call
  // (epic_last_kernel_times): kev[i] .. kev[i + 1] is kernel i
  cudaEvent_t kev[4] = {nullptr, nullptr, nullptr, nullptr};
  int nk = 0;
  const char* kname[3] = {nullptr, nullptr, nullptr};
  // the same around the two kernels of the last epic_select_compatible_subset
  cudaEvent_t sev[3] = {nullptr, nullptr, nullptr};
  bool sel_timed = false;
};

namespace {
// record event i of the table's kernel timing on st (created on first use)
void mark_event(cudaEvent_t* e, cudaStream_t st) {
  if (!*e && cudaEventCreate(e) != cudaSuccess) *e = nullptr;
  if (*e) cudaEventRecord(*e, st);
}
void mark(epic_lexer_table* t, int i, cudaStream_t st) { mark_event(&t->kev[i], st); }
}  // namespace

namespace {

template <class T>
epic_status upload(epic_grammar* g, const std::vector<T>& v, const T** out) {
  void* p = nullptr;
  size_t bytes = std::max<size_t>(sizeof(T), v.size() * sizeof(T));
  if (cudaMalloc(&p, bytes) != cudaSuccess) return EPIC_ERR_OOM;
  g->dev_allocs.push_back(p);
  if (!v.empty() && cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess)
    return EPIC_ERR_CUDA;
  *out = (const T*)p;
  return EPIC_OK;
}

// Device memory for a workspace; false (and no error left behind for the next
// call's check of its launches) when there is not enough.
template <class T>
bool device_alloc(T** p, size_t bytes) {
  if (cudaMalloc((void**)p, bytes) == cudaSuccess) return true;
  (void)cudaGetLastError();
  *p = nullptr;
  return false;
}

// The workspaces in use now belong to a graph if `st` is being captured.
// Called before a call's launches.
epic_status note_capture(epic_lexer_table* t, cudaStream_t st) {
  if (!st) return EPIC_OK;  // the legacy stream cannot be captured
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) return EPIC_ERR_CUDA;
  if (cap != cudaStreamCaptureStatusActive) return EPIC_OK;
  try {
    for (void* p : {(void*)t->d_ws, (void*)t->d_wws, (void*)t->d_spec, (void*)t->d_seq, (void*)t->d_regs, (void*)t->d_wit})
      if (p && std::find(t->in_graphs.begin(), t->in_graphs.end(), p) == t->in_graphs.end()) t->in_graphs.push_back(p);
  } catch (std::exception&) {
    return EPIC_ERR_OOM;
  }
  return EPIC_OK;
}

// Give a workspace back (after the table's last stream), unless a graph holds it.
template <class T>
void release(epic_lexer_table* t, T** p) {
  if (*p && std::find(t->in_graphs.begin(), t->in_graphs.end(), (void*)*p) == t->in_graphs.end()) {
    cudaStreamSynchronize(t->last);
    cudaFree(*p);
  }
  *p = nullptr;
}

int sm_count() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

// Default budget of one device workspace: a share of the GPU's memory, and no
// more than it holds already plus what is free now less 1 GiB of headroom (so
// a call that ran once finds the same room again).  An environment variable (MiB)
// overrides.  The three workspaces (per-sequence charts 30 %, warp walks
// 25 %, block walks 25 %) leave a fifth of the GPU to the caller.
size_t workspace_budget(const char* env, double share, size_t held) {
  if (const char* e = getenv(env)) return strtoull(e, nullptr, 10) << 20;
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return (size_t)4096 << 20;
  const size_t headroom = (size_t)1 << 30;
  return std::min((size_t)(share * (double)total_b), held + (free_b > headroom ? free_b - headroom : 0));
}

// Block-walk workspace of selection, the fallback and few checks: every CTA
// gets room for one whole chart of a row (4,096 columns, 640 n entries, as the
// per-sequence forward charts; EPIC_ENTRIES_PER_CTA overrides), and as many
// CTAs as asked run if their workspaces fit EPIC_WORKSPACE_MB (default a
// quarter of the GPU), else fewer (the kernels loop over their sequences).
struct BlockPlan {
  WsDims d;
  size_t per;
  int ctas;
};
BlockPlan plan_workspace(const epic_lexer_table* t, int want_ctas, int n) {
  const epic_grammar* g = t->g;
  int W = g->dg.W, VW = g->dg.VW, FW = g->dg.FW;
  BlockPlan p;
  WsDims& d = p.d;
  d.nmax = kMaxCols;
  d.emax = std::max<long long>(4096, 640ll * std::max(1, n));
  if (const char* e = getenv("EPIC_ENTRIES_PER_CTA")) d.emax = std::max<long long>(64, atoll(e));
  const size_t budget = workspace_budget("EPIC_WORKSPACE_MB", 0.25, t->d_ws ? t->ws_bytes : 0);
  p.per = ws_bytes_per_cta(d, W, VW, FW);
  while (p.per > budget && d.emax > 4096) {  // not even one CTA fits: smaller charts
    d.emax = d.emax * 3 / 4;
    p.per = ws_bytes_per_cta(d, W, VW, FW);
  }
  p.ctas = (int)std::max<long long>(1, std::min<long long>(std::max(1, want_ctas), (long long)(budget / p.per)));
  return p;
}
epic_status ensure_workspace(epic_lexer_table* t, const BlockPlan& p, cudaStream_t st) {
  const WsDims d = p.d;
  const int ctas = p.ctas;
  const size_t need = p.per * (size_t)ctas;
  if (t->d_ws && t->ws_bytes >= need && t->dims.nmax == d.nmax && t->dims.emax == d.emax) {
    t->ctas = ctas;
    return EPIC_OK;
  }
  release(t, &t->d_ws);
  if (!device_alloc(&t->d_ws, need)) return EPIC_ERR_OOM;
  // staging rows and bdone must start at zero; the rest is written before read
  if (cudaMemsetAsync(t->d_ws, 0, need, st) != cudaSuccess) return EPIC_ERR_CUDA;
  t->ws_bytes = need;
  t->dims = d;
  t->ctas = ctas;
  return EPIC_OK;
}

// Chart entries of a whole walk of validation.
long long walk_entries(int n) {
  if (const char* e = getenv("EPIC_ENTRIES_PER_WALK")) return atoll(e);
  return 256ll * std::max(1, n);
}

// Warp-walk workspace: columns <= min(4096, 8 n + 256) per walk; entries
// per walk EPIC_ENTRIES_PER_WALK (default 256 n); warps cut down until the
// total fits EPIC_WARP_WORKSPACE_MB (default a quarter of the GPU).
epic_status ensure_wworkspace(epic_lexer_table* t, long long checks, int n, cudaStream_t st) {
  const epic_grammar* g = t->g;
  int W = g->dg.W;
  int nmax = std::min(kWCols, 8 * n + 256);
  const long long emax = walk_entries(n);
  const size_t budget = workspace_budget("EPIC_WARP_WORKSPACE_MB", 0.25, t->d_wws ? t->wws_bytes : 0);
  size_t per = wbytes_per_warp(nmax, emax, W);
  long long warps = std::min<long long>(checks, (long long)sm_count() * 2 * kWarpsPerCta);
  warps = std::max<long long>(kWarpsPerCta, (warps + kWarpsPerCta - 1) / kWarpsPerCta * kWarpsPerCta);
  while (warps > kWarpsPerCta && per * (size_t)warps > budget) warps -= kWarpsPerCta;
  size_t need = per * (size_t)warps;
  if (t->d_wws && t->wws_bytes >= need && t->wnmax == nmax && t->wemax == emax) {
    t->wwarps = (int)std::min<long long>(warps, t->wws_bytes / per / kWarpsPerCta * kWarpsPerCta);
    return EPIC_OK;
  }
  release(t, &t->d_wws);
  if (!device_alloc(&t->d_wws, need)) return EPIC_ERR_OOM;
  if (cudaMemsetAsync(t->d_wws, 0, need, st) != cudaSuccess) return EPIC_ERR_CUDA;
  t->wws_bytes = need;
  t->wnmax = nmax;
  t->wemax = emax;
  t->wwarps = (int)warps;
  return EPIC_OK;
}

WPack wpack_of(const epic_lexer_table* t) {
  WPack p;
  p.base = t->d_wws;
  p.nmax = t->wnmax;
  p.emax = t->wemax;
  p.W = t->g->dg.W;
  p.per_warp = wbytes_per_warp(p.nmax, p.emax, p.W);
  return p;
}

// Grow a device buffer owned by the table (synchronizing its last stream first).
epic_status grow(epic_lexer_table* t, char** buf, size_t* have, size_t need) {
  if (*buf && *have >= need) return EPIC_OK;
  release(t, buf);
  *have = 0;
  if (!device_alloc(buf, need)) return EPIC_ERR_OOM;
  *have = need;
  return EPIC_OK;
}

// Checks by region, steps 1-2 (also the start of witness extraction): the
// per-sequence arena (EPIC_SEQ_ENTRIES, default 640 n chart entries per
// sequence; EPIC_SEQ_WORKSPACE_MB, default 30 % of the GPU, caps the batch:
// a sequence whose chart does not fit its arena has its checks walk the
// whole graph instead), the forward charts and the good masks with their
// indexes.
epic_status region_prepare(const epic_grammar* g, epic_lexer_table* t, const int32_t* d_x, int B, int n, SeqPack& sp,
                           cudaStream_t st) {
  (void)g;
  const DevGrammar& dg = t->dgl;
  sp.nmax = std::min(kMaxCols, 8 * n + 256);
  sp.n = n;
  sp.W = dg.W;
  sp.VW = dg.VW;
  sp.edge_cap = 32 * sp.nmax;
  sp.emax = 640ll * n;
  if (const char* e = getenv("EPIC_SEQ_ENTRIES")) sp.emax = atoll(e);
  const size_t budget = workspace_budget("EPIC_SEQ_WORKSPACE_MB", 0.30, t->d_seq ? t->seq_bytes : 0);
  while (sp.emax > 4096 && sp.bytes() * (size_t)B > budget) sp.emax = sp.emax * 3 / 4;
  sp.per_seq = sp.bytes();
  epic_status s = grow(t, &t->d_seq, &t->seq_bytes, sp.per_seq * (size_t)B);
  if (s != EPIC_OK) return s;
  sp.base = t->d_seq;
  s = note_capture(t, st);
  if (s != EPIC_OK) return s;
  t->last = st;
  // 1. forward charts
  {
    t->nk = 3;
    t->kname[0] = "k_forward_gs";
    t->kname[1] = "k_good";
    t->kname[2] = "k_check";
    mark(t, 0, st);
    launch_forward_gs(std::min(B, 4 * sm_count()), st, dg, t->d_table, t->vocab, d_x, B, n, sp, t->d_stats);
  }
  // 2. good masks
  mark(t, 1, st);
  launch_good(B, st, dg, sp);
  mark(t, 2, st);
  return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

epic_status validate_region(const epic_grammar* g, epic_lexer_table* t, const int32_t* d_x, int B, int n,
                            const int32_t* d_pos, int k, const int32_t* d_cand, int K, uint8_t* d_valid,
                            cudaStream_t st) {
  const DevGrammar& dg = t->dgl;
  long long total = (long long)B * k * K;
  // per-warp workspace of the checks: own columns after the chart's
  WPack wp;
  wp.nmax = kWCols;
  // own entries: the region's columns and the rows carried after it (narrow
  // rows: as much as a whole walk, since a region can be most of a row)
  wp.emax = std::max(8192ll, (dg.W <= 32 ? 256ll : 64ll) * n);
  if (const char* e = getenv("EPIC_ENTRIES_PER_WALK")) wp.emax = atoll(e);
  wp.W = dg.W;
  wp.per_warp = wbytes_per_warp(wp.nmax, wp.emax, wp.W);
  const size_t wbudget = workspace_budget("EPIC_WARP_WORKSPACE_MB", 0.25, t->d_wws ? t->wws_bytes : 0);
  long long warps = std::min<long long>(total, (long long)sm_count() * 2 * kWarpsPerCta);
  warps = std::max<long long>(1, warps);
  warps = std::max<long long>(1, std::min<long long>(warps, (long long)(wbudget / wp.per_warp)));
  size_t wneed = wp.per_warp * (size_t)warps;
  if (!t->d_wws || t->wws_bytes < wneed || t->wnmax != wp.nmax || t->wemax != wp.emax) {
    release(t, &t->d_wws);
    if (!device_alloc(&t->d_wws, wneed)) return EPIC_ERR_OOM;
    // the global stage starts at zero; walks return it zeroed
    if (cudaMemsetAsync(t->d_wws, 0, wneed, st) != cudaSuccess) return EPIC_ERR_CUDA;
    t->wws_bytes = wneed;
    t->wnmax = wp.nmax;
    t->wemax = wp.emax;
  }
  wp.base = t->d_wws;
  epic_status s = grow(t, (char**)&t->d_regs, &t->regs_bytes, (size_t)warps * 3 * wp.nmax * 4);
  if (s != EPIC_OK) return s;
  t->last = st;
  // 1-2. forward charts and good masks
  SeqPack sp;
  s = region_prepare(g, t, d_x, B, n, sp, st);
  if (s != EPIC_OK) return s;
  t->n_region += total;
  t->n_vkernels += 3;
  // 3. checks
  cudaMemsetAsync(t->d_counter, 0, 8, st);
  const int per_cta = (int)std::min<long long>(kWarpsPerCta, warps);  // every warp owns an allocated workspace
  launch_check((int)std::max<long long>(1, warps / per_cta), 32 * per_cta, st, dg, t->d_table, t->vocab, d_x, n, d_pos,
               k, d_cand, K, total, d_valid, sp, wp, t->d_regs, t->d_counter, t->d_stats);
  mark(t, 3, st);
  return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

// Whole-graph walks with a CTA per check (`slots` of them at a time) or with a
// warp per check?  A CTA walk ends several times sooner and fills an SM, so it
// wins while every check has a slot at once (ms with a CTA / a warp / by
// region): JSON 4 x 64, 128 checks 1.8 / 2.9 / 3.0; molecules 4 x 96, 128
// checks 6.2 / 18 / 12.  Two rounds of 96 tokens and more, 256 checks: molecules
// 4 x 96 13 / 22 / 19, 16 x 120 16 / 33 / 21, 2 x 200 32 / 81 / 42; about even
// on JSON, 4 x 100 5.0 / 4.5 / 6.0, 16 x 100 5.0 / 6.6 / 6.0, 2 x 200 11 / 13 /
// 11, 1 x 256 12.5 / 10.1 / 10.9.  Shorter rows lose then (JSON 4 x 64 3.2 / 2.3
// / 3.4).  Grammars of at most 4 item words have too little in a column
// (expressions 4 x 32, 32 checks 1.06 / 1.07).
bool cta_walks(long long total, int n, int W, long long slots) {
  if (W <= 4) return false;
  return total <= slots || (W <= 32 && n >= 96 && total <= 2 * slots);
}

WsPack pack_of(const epic_lexer_table* t) {
  WsPack p;
  p.base = t->d_ws;
  p.dims = t->dims;
  p.W = t->g->dg.W;
  p.VW = t->g->dg.VW;
  p.FW = t->g->dg.FW;
  p.per_cta = ws_bytes_per_cta(t->dims, p.W, p.VW, p.FW);
  return p;
}

}  // namespace

extern "C" {

#ifdef EPIC_PHASE_TIMERS
// measurement build only: per-phase cycle counters (the walks' and the GS
// columns' in out16, the good pass's in out16 + 16)
int epic_debug_phase_read(unsigned long long* out16, int reset) {
  if (cudaDeviceSynchronize() != cudaSuccess) return -1;
  for (int i = 0; i < 16; ++i) out16[i] = 0;
  if (phase_read_walk(out16, reset) != 0 || phase_read_forward(out16, reset) != 0 ||
      phase_read_check(out16, reset) != 0)
    return -1;
  for (int i = 0; i < 16; ++i) out16[16 + i] = 0;
  if (phase_read_good(out16 + 16, reset) != 0) return -1;
  return 0;
}
#endif

const char* epic_status_string(epic_status s) {
  switch (s) {
    case EPIC_OK: return "ok";
    case EPIC_ERR_INVALID_ARG: return "invalid argument";
    case EPIC_ERR_GRAMMAR: return "invalid grammar (malformed or empty language)";
    case EPIC_ERR_LEXER: return "invalid lexer specification";
    case EPIC_ERR_OOM: return "out of memory";
    case EPIC_ERR_CUDA: return "CUDA error";
    case EPIC_ERR_CAPACITY: return "capacity exceeded";
    case EPIC_ERR_TIMEOUT: return "device loop bound exceeded";
  }
  return "unknown status";
}

epic_status epic_grammar_create(const epic_grammar_desc* desc, epic_grammar** out) {
  if (!desc || !out) return EPIC_ERR_INVALID_ARG;
  *out = nullptr;
  if (desc->n_terminals <= 0 || desc->n_terminals > 255 || desc->n_nonterminals <= 0 ||
      desc->n_nonterminals > 32 * kMaxVW || desc->n_productions < 0 || !desc->terminal_regex ||
      !desc->terminal_skip || (desc->n_productions > 0 && (!desc->lhs || !desc->rhs_off)))
    return EPIC_ERR_INVALID_ARG;
  int dev_count = 0;
  if (cudaGetDeviceCount(&dev_count) != cudaSuccess || dev_count == 0) return EPIC_ERR_CUDA;
  epic_grammar* g = new (std::nothrow) epic_grammar();
  if (!g) return EPIC_ERR_OOM;
  cudaGetDevice(&g->device);
  int T = desc->n_terminals, V = desc->n_nonterminals, P = desc->n_productions;
  try {
    std::vector<std::string> rx;
    for (int t = 0; t < T; ++t) {
      if (!desc->terminal_regex[t]) throw std::invalid_argument("null regex");
      rx.emplace_back(desc->terminal_regex[t]);
    }
    try {
      g->dfa = build_lexer(rx);
    } catch (std::runtime_error&) {
      delete g;
      return EPIC_ERR_LEXER;
    }
    if (g->dfa.Q > kMaxQ) {
      delete g;
      return EPIC_ERR_CAPACITY;
    }
    std::vector<uint8_t> skip(desc->terminal_skip, desc->terminal_skip + T);
    std::vector<int32_t> lhs(desc->lhs, desc->lhs + P);
    std::vector<int32_t> off(desc->rhs_off, desc->rhs_off + P + 1);
    if (off[0] != 0) throw std::invalid_argument("rhs_off[0] != 0");
    std::vector<int32_t> rhs;
    if (off[P] > 0) {
      if (!desc->rhs) throw std::invalid_argument("null rhs");
      rhs.assign(desc->rhs, desc->rhs + off[P]);
    }
    try {
      g->tabs = build_tables(T, skip, V, desc->start, lhs, off, rhs);
    } catch (std::domain_error&) {
      delete g;
      return EPIC_ERR_GRAMMAR;
    }
  } catch (std::exception&) {
    delete g;
    return EPIC_ERR_INVALID_ARG;
  }
  GrammarTables& G = g->tabs;
  if (G.W > kMaxW) {
    delete g;
    return EPIC_ERR_CAPACITY;
  }
  g->cov = build_cover(G);
  if (g->cov.FW > kMaxFW) {
    delete g;
    return EPIC_ERR_CAPACITY;
  }
  DevGrammar& d = g->dg;
  d.T = G.T;
  d.V = G.V;
  d.D = G.D;
  d.W = G.W;
  d.VW = (G.V + 31) / 32;
  d.Q = g->dfa.Q;
  d.start_item = G.start_item;
  d.accept_item = G.accept_item;
  std::vector<uint32_t> next_any(G.W);
  for (int w = 0; w < G.W; ++w) next_any[w] = G.any_term[w] | G.any_nt[w];
  std::vector<int16_t> inext(G.D), ilhs(G.D);
  for (int i = 0; i < G.D; ++i) {
    inext[i] = (int16_t)G.item_next[i];
    ilhs[i] = (int16_t)G.item_lhs[i];
  }
  epic_status st = EPIC_OK;
  auto up = [&](auto& v, auto** o) {
    if (st == EPIC_OK) st = upload(g, v, o);
  };
  up(G.exp_term, &d.exp_term);
  up(G.exp_nt, &d.exp_nt);
  up(G.any_nt, &d.any_nt);
  up(G.any_term, &d.any_term);
  up(next_any, &d.next_any);
  up(G.nullable_next, &d.nullable_next);
  up(G.complete, &d.complete);
  up(G.pred, &d.pred);
  up(G.gap_pred, &d.gap_pred);
  up(G.follow, &d.follow);
  {
    std::vector<int16_t> nt((size_t)32 * G.W, -1);
    for (int i = 0; i < G.D; ++i)
      if (G.item_next[i] >= G.T) nt[(size_t)(i & 31) * G.W + (i >> 5)] = (int16_t)(G.item_next[i] - G.T);
    up(nt, &d.next_t);
  }
  up(inext, &d.item_next);
  up(ilhs, &d.item_lhs);
  up(g->dfa.accept, &d.dfa_accept);
  up(g->dfa.next, &d.dfa_next);
  std::vector<uint8_t> ext(g->dfa.Q, 0);
  for (int q = 0; q < g->dfa.Q; ++q)
    for (int c = 0; c < 256; ++c)
      if (g->dfa.next[(size_t)q * 256 + c] >= 0) ext[q] = 1;
  up(ext, &d.dfa_ext);
  up(G.skip, &d.skip);
  {
    // complete / waiting items by nonterminal as (word, mask) pairs
    auto lists = [&](auto member, std::vector<int32_t>& off, std::vector<uint2>& lst) {
      std::vector<std::vector<uint2>> by((size_t)G.V);
      for (int i = 0; i < G.D; ++i) {
        const int A = member(i);
        if (A < 0) continue;
        auto& l = by[(size_t)A];
        if (l.empty() || l.back().x != (uint32_t)(i >> 5)) l.push_back(uint2{(uint32_t)(i >> 5), 0u});
        l.back().y |= 1u << (i & 31);
      }
      off.assign(1, 0);
      for (auto& l : by) {
        lst.insert(lst.end(), l.begin(), l.end());
        off.push_back((int32_t)lst.size());
      }
    };
    std::vector<int32_t> coff, woff;
    std::vector<uint2> cl, wl;
    lists([&](int i) { return G.item_next[i] < 0 && i != G.accept_item ? G.item_lhs[i] : -1; }, coff, cl);
    lists([&](int i) { return G.item_next[i] >= G.T ? G.item_next[i] - G.T : -1; }, woff, wl);
    d.n_cpl = (int)cl.size();
    d.n_wait = (int)wl.size();
    std::vector<uint2> w4((size_t)G.V, uint2{0u, 0u});
    std::vector<uint4> m4((size_t)G.V, uint4{0u, 0u, 0u, 0u});
    for (int A = 0; A < G.V; ++A) {
      uint32_t* m = &m4[(size_t)A].x;
      for (int q = coff[A], j = 0; q < coff[A + 1]; ++q, ++j) {
        if (j == 4) {
          w4[(size_t)A].y = 1u;
          break;
        }
        w4[(size_t)A].x |= cl[(size_t)q].x << (8 * j);
        m[j] = cl[(size_t)q].y;
      }
    }
    up(w4, &d.cpl4w);
    up(m4, &d.cpl4m);
    up(coff, &d.cpl_off);
    up(cl, &d.cpl);
    up(woff, &d.wait_off);
    up(wl, &d.wait);
    d.any_nullable = 0;
    for (uint32_t m : G.nullable_next) d.any_nullable |= m != 0;
  }
  {
    // runs of advanceable items for the doubling closure (see device.cuh)
    int maxlen = 0;
    for (size_t p = 0; p + 1 < G.rhs_off.size(); ++p) maxlen = std::max(maxlen, G.rhs_off[p + 1] - G.rhs_off[p]);
    int steps = 1;
    while ((1 << steps) <= maxlen) ++steps;
    d.adv_steps = steps;
    std::vector<uint32_t> pw((size_t)2 * steps * G.W, 0);
    auto bit = [&](const std::vector<uint32_t>& m, long long i) -> bool {
      return i >= 0 && i < (long long)G.W * 32 && ((m[(size_t)(i >> 5)] >> (i & 31)) & 1u);
    };
    for (int mode = 0; mode < 2; ++mode) {
      std::vector<uint32_t> cur = mode ? next_any : G.nullable_next;
      for (int st2 = 0; st2 < steps; ++st2) {
        std::copy(cur.begin(), cur.end(), pw.begin() + ((size_t)mode * steps + st2) * G.W);
        const long long k = 1ll << st2;  // next: i and i + k both start runs of length k
        std::vector<uint32_t> nx(G.W, 0);
        for (long long i = 0; i < (long long)G.W * 32; ++i)
          if (bit(cur, i) && bit(cur, i + k)) nx[(size_t)(i >> 5)] |= 1u << (i & 31);
        cur.swap(nx);
      }
    }
    up(pw, &d.adv_pow);
  }
  {
    // witness extraction tables: complete items by left side, and a shortest
    // terminal string of every nonterminal (fixpoint of the shortest yield
    // length; a production is chosen only when it strictly shortens, so the
    // choices form no cycle and expand to finite strings)
    const int V = G.V, T = G.T;
    const int P2 = (int)G.lhs.size();
    std::vector<int32_t> coff(V + 1, 0), citems;
    for (int p = 0; p < P2; ++p)
      if (G.lhs[p] >= 0) ++coff[G.lhs[p] + 1];
    for (int v = 0; v < V; ++v) coff[v + 1] += coff[v];
    citems.assign(coff[V], 0);
    std::vector<int32_t> cur(coff.begin(), coff.end() - 1);
    for (int p = 0; p < P2; ++p)
      if (G.lhs[p] >= 0) citems[cur[G.lhs[p]]++] = G.item_base[p] + (G.rhs_off[p + 1] - G.rhs_off[p]);
    const long long INF = 1ll << 40;
    std::vector<long long> len(V, INF);
    std::vector<int> best(V, -1);
    for (bool changed = true; changed;) {
      changed = false;
      for (int p = 0; p < P2; ++p) {
        if (G.lhs[p] < 0) continue;
        long long L = 0;
        for (int i = G.rhs_off[p]; i < G.rhs_off[p + 1] && L < INF; ++i) {
          const int X = G.rhs[i];
          L += X < T ? 1 : len[X - T];
        }
        if (L < len[G.lhs[p]]) {
          len[G.lhs[p]] = L;
          best[G.lhs[p]] = p;
          changed = true;
        }
      }
    }
    std::vector<int32_t> yoff(V + 1, 0), ys;
    std::vector<std::vector<int32_t>> memo(V);
    std::vector<char> done(V, 0);
    std::function<void(int, std::vector<int32_t>&)> expand = [&](int A, std::vector<int32_t>& out) {
      if (done[A]) {
        out.insert(out.end(), memo[A].begin(), memo[A].end());
        return;
      }
      std::vector<int32_t> mine;
      const int p = best[A];
      if (p >= 0 && mine.size() < 4096)
        for (int i = G.rhs_off[p]; i < G.rhs_off[p + 1]; ++i) {
          const int X = G.rhs[i];
          if (X < T) mine.push_back(X);
          else expand(X - T, mine);
        }
      if (mine.size() > 4096) mine.resize(4096);
      memo[A] = mine;
      done[A] = 1;
      out.insert(out.end(), mine.begin(), mine.end());
    };
    for (int v = 0; v < V; ++v) {
      std::vector<int32_t> y;
      if (len[v] < INF) expand(v, y);
      yoff[v + 1] = yoff[v] + (int)y.size();
      ys.insert(ys.end(), y.begin(), y.end());
    }
    up(coff, &d.nt_comp_off);
    up(citems, &d.nt_comp);
    up(yoff, &d.ny_off);
    up(ys, &d.ny);
  }
  d.FS = g->cov.FS;
  d.FW = g->cov.FW;
  d.cov_start = g->cov.start;
  d.cov_accept = g->cov.accept;
  up(g->cov.eps_close, &d.cov_eps_close);
  up(g->cov.all_close, &d.cov_all_close);
  if (st != EPIC_OK) {
    epic_grammar_destroy(g);
    return st;
  }
  *out = g;
  return EPIC_OK;
}

void epic_grammar_destroy(epic_grammar* g) {
  if (!g) return;
  for (void* p : g->dev_allocs) cudaFree(p);
  delete g;
}

int32_t epic_grammar_lexer_states(const epic_grammar* g) { return g ? g->dfa.Q : -1; }

epic_status epic_lexer_table_build(const epic_grammar* g, const int32_t* tok_off, const uint8_t* tok_bytes,
                                   int32_t vocab, void* cuda_stream, epic_lexer_table** out) {
  if (!g || !tok_off || !out || vocab <= 0) return EPIC_ERR_INVALID_ARG;
  *out = nullptr;
  if (tok_off[0] != 0) return EPIC_ERR_INVALID_ARG;
  for (int t = 0; t < vocab; ++t) {
    int L = tok_off[t + 1] - tok_off[t];
    if (L < 1 || L > 64) return EPIC_ERR_INVALID_ARG;
  }
  if (!tok_bytes) return EPIC_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  epic_lexer_table* t = new (std::nothrow) epic_lexer_table();
  if (!t) return EPIC_ERR_OOM;
  t->g = g;
  t->vocab = vocab;
  t->last = st;
  t->dgl = g->dg;
  t->dgl.lazy = LazyLex{};
  int Q = g->dg.Q;
  size_t nbytes = (size_t)tok_off[vocab];
  int32_t* d_off = nullptr;
  uint8_t* d_bytes = nullptr;
  int* d_ovf = nullptr;
  epic_status res = EPIC_OK;
  if (cudaMalloc(&t->d_table, (size_t)vocab * Q * sizeof(LexEntry)) != cudaSuccess ||
      cudaMalloc(&d_off, (size_t)(vocab + 1) * 4) != cudaSuccess || cudaMalloc(&d_bytes, nbytes) != cudaSuccess ||
      cudaMalloc(&d_ovf, 4) != cudaSuccess || cudaMalloc(&t->d_stats, S_N * 8) != cudaSuccess ||
      cudaMalloc(&t->d_counter, 8) != cudaSuccess) {
    res = EPIC_ERR_OOM;
  }
  if (res == EPIC_OK) {
    cudaMemcpyAsync(d_off, tok_off, (size_t)(vocab + 1) * 4, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(d_bytes, tok_bytes, nbytes, cudaMemcpyHostToDevice, st);
    cudaMemsetAsync(d_ovf, 0, 4, st);
    cudaMemsetAsync(t->d_stats, 0, S_N * 8, st);
    long long total = (long long)vocab * Q;
    int threads = 256;
    long long blocks = (total + threads - 1) / threads;
    k_lex_table<<<(unsigned)blocks, threads, 0, st>>>(d_off, d_bytes, vocab, Q, g->dg.dfa_next, g->dg.dfa_accept,
                                                       g->dg.skip, t->d_table, d_ovf);
    int ovf = 0;
    if (cudaGetLastError() != cudaSuccess || cudaMemcpyAsync(&ovf, d_ovf, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      res = EPIC_ERR_CUDA;
    else if (ovf)
      res = EPIC_ERR_CAPACITY;
  }
  cudaFree(d_off);
  cudaFree(d_bytes);
  cudaFree(d_ovf);
  if (res != EPIC_OK) {
    epic_lexer_table_destroy(t);
    return res;
  }
  t->dgl.lazy.stats = t->d_stats + S_LEX_LOOKUPS;  // lookups are counted for dense tables too
  *out = t;
  return EPIC_OK;
}

epic_status epic_lexer_table_build_lazy(const epic_grammar* g, const int32_t* tok_off, const uint8_t* tok_bytes,
                                        int32_t vocab, int64_t capacity, void* cuda_stream, epic_lexer_table** out) {
  if (!g || !tok_off || !out || vocab <= 0 || capacity < 1) return EPIC_ERR_INVALID_ARG;
  *out = nullptr;
  if (tok_off[0] != 0) return EPIC_ERR_INVALID_ARG;
  for (int t = 0; t < vocab; ++t) {
    int L = tok_off[t + 1] - tok_off[t];
    if (L < 1 || L > 64) return EPIC_ERR_INVALID_ARG;
  }
  if (!tok_bytes) return EPIC_ERR_INVALID_ARG;
  // the key token * Q + state + 1 must fit 32 bits
  if ((unsigned long long)vocab * (unsigned long long)g->dg.Q >= 0xFFFFFFFFull) return EPIC_ERR_CAPACITY;
  long long cap = 1;
  while (cap < capacity) cap <<= 1;
  if (cap > (1ll << 30)) return EPIC_ERR_CAPACITY;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  epic_lexer_table* t = new (std::nothrow) epic_lexer_table();
  if (!t) return EPIC_ERR_OOM;
  t->g = g;
  t->vocab = vocab;
  t->last = st;
  t->lz_cap = cap;
  size_t nbytes = (size_t)tok_off[vocab];
  epic_status res = EPIC_OK;
  if (cudaMalloc(&t->d_lz_keys, (size_t)cap * 4) != cudaSuccess ||
      cudaMalloc(&t->d_lz_ready, (size_t)cap * 4) != cudaSuccess ||
      cudaMalloc(&t->d_lz_vals, (size_t)cap * sizeof(LexEntry)) != cudaSuccess ||
      cudaMalloc(&t->d_lz_off, (size_t)(vocab + 1) * 4) != cudaSuccess ||
      cudaMalloc(&t->d_lz_bytes, nbytes) != cudaSuccess || cudaMalloc(&t->d_stats, S_N * 8) != cudaSuccess ||
      cudaMalloc(&t->d_counter, 8) != cudaSuccess)
    res = EPIC_ERR_OOM;
  if (res == EPIC_OK) {
    cudaMemcpyAsync(t->d_lz_off, tok_off, (size_t)(vocab + 1) * 4, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(t->d_lz_bytes, tok_bytes, nbytes, cudaMemcpyHostToDevice, st);
    cudaMemsetAsync(t->d_lz_keys, 0, (size_t)cap * 4, st);
    cudaMemsetAsync(t->d_lz_ready, 0, (size_t)cap * 4, st);
    cudaMemsetAsync(t->d_stats, 0, S_N * 8, st);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) res = EPIC_ERR_CUDA;
  }
  if (res != EPIC_OK) {
    epic_lexer_table_destroy(t);
    return res;
  }
  t->dgl = g->dg;
  t->dgl.lazy.keys = t->d_lz_keys;
  t->dgl.lazy.ready = t->d_lz_ready;
  t->dgl.lazy.vals = t->d_lz_vals;
  t->dgl.lazy.mask = (uint32_t)(cap - 1);
  t->dgl.lazy.tok_off = t->d_lz_off;
  t->dgl.lazy.tok_bytes = t->d_lz_bytes;
  t->dgl.lazy.stats = t->d_stats + S_LEX_LOOKUPS;
  *out = t;
  return EPIC_OK;
}

void epic_lexer_table_destroy(epic_lexer_table* t) {
  if (!t) return;
  if (t->last) cudaStreamSynchronize(t->last);
  release(t, &t->d_ws);
  release(t, &t->d_wws);
  release(t, &t->d_spec);
  release(t, &t->d_seq);
  release(t, &t->d_regs);
  release(t, &t->d_wit);
  for (void* p : t->in_graphs) cudaFree(p);
  cudaFree(t->d_table);
  cudaFree(t->d_fb);
  cudaFree(t->d_stats);
  cudaFree(t->d_counter);
  cudaFree(t->d_lz_keys);
  cudaFree(t->d_lz_ready);
  cudaFree(t->d_lz_vals);
  cudaFree(t->d_lz_off);
  cudaFree(t->d_lz_bytes);
  for (cudaEvent_t e : t->kev)
    if (e) cudaEventDestroy(e);
  for (cudaEvent_t e : t->sev)
    if (e) cudaEventDestroy(e);
  delete t;
}

epic_status epic_lexer_table_copy(const epic_lexer_table* t, int32_t first_token, int32_t count, void* host_out,
                                  size_t out_bytes) {
  if (!t || !host_out || first_token < 0 || count < 0 || first_token + count > t->vocab || !t->d_table)
    return EPIC_ERR_INVALID_ARG;
  size_t Q = (size_t)t->g->dg.Q;
  size_t bytes = (size_t)count * Q * sizeof(LexEntry);
  if (out_bytes < bytes) return EPIC_ERR_INVALID_ARG;
  if (cudaStreamSynchronize(t->last) != cudaSuccess) return EPIC_ERR_CUDA;
  if (cudaMemcpy(host_out, t->d_table + (size_t)first_token * Q, bytes, cudaMemcpyDeviceToHost) != cudaSuccess)
    return EPIC_ERR_CUDA;
  return EPIC_OK;
}

epic_status epic_validate_batch(const epic_grammar* g, const epic_lexer_table* tc, const int32_t* d_x, int32_t B,
                                int32_t n, const int32_t* d_pos, int32_t k, const int32_t* d_cand, int32_t K,
                                uint8_t* d_valid, void* cuda_stream) {
  epic_lexer_table* t = const_cast<epic_lexer_table*>(tc);
  if (!g || !t || t->g != g || B < 0 || n < 0 || k < 0 || K < 0) return EPIC_ERR_INVALID_ARG;
  long long total = (long long)B * k * K;
  if (total == 0) return EPIC_OK;
  if (!d_x || !d_pos || !d_cand || !d_valid || n == 0) return EPIC_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  // Few checks of narrow item sets walk their whole graphs, a CTA each.  Else
  // checks by region over a per-sequence chart, built once per sequence
  // instead of once per check: when the item sets are wide (a warp takes
  // seconds for a long row of a large grammar), when there are more checks
  // than resident walks, and on rows of at least 128 tokens.  By region
  // against a warp per check, 1,024 checks of JSON: 16 x 64 4.0 against 3.1 ms,
  // 16 x 128 8.4 against 6.7, 16 x 256 24 against 33; expressions (two words):
  // 1 x 128, 64 checks 10.9 against 7.2, 1 x 256 26 against 30, 16 x 256 35
  // against 41.  The lines cross between 128 and 256 tokens; 128 keeps the
  // longer walks off the warps.
  // Wide item sets go by region however few the checks, and region_checks
  // counts them so.  (A CTA each would end sooner for a handful: C-like 1 x 48,
  // 32 checks 3.7 ms against 7.3; 400 nonterminals 1 x 256, 16 checks 188
  // against 282, 1 x 1024, 4 checks 12.0 s against 13.5.)
  bool few = g->dg.W <= 32 && cta_walks(total, n, g->dg.W, sm_count());
  bool region = !few && (g->dg.W > 32 || n >= 128 || total > (long long)sm_count() * 2 * kWarpsPerCta);
  bool forced = false;
  if (const char* e = getenv("EPIC_REGION")) {
    region = atoi(e) != 0;
    few = few && !region;
    forced = region;
  }
  if (region) {
    const epic_status s = validate_region(g, t, d_x, B, n, d_pos, k, d_cand, K, d_valid, st);
    // narrow item sets take this way for speed only: without memory for the
    // charts, a warp walks each check (nothing was launched)
    if (s != EPIC_ERR_OOM || g->dg.W > 32 || forced) return s;
  }
  // Few checks: a CTA each, where the block workspace holds a slot for each
  // and charts as large as a warp's (a tight budget: a warp each).
  const int slots = (int)std::min<long long>(total, sm_count());
  if (few) {
    const BlockPlan p = plan_workspace(t, slots, n);
    few = p.ctas == slots && p.d.emax >= walk_entries(n);
    if (few) {
      const epic_status s = ensure_workspace(t, p, st);
      if (s != EPIC_OK && s != EPIC_ERR_OOM) return s;
      few = s == EPIC_OK;
    }
  }
  if (few) {
    long long cap = t->dims.emax;
    if (const char* e = getenv("EPIC_ENTRIES_PER_WALK")) cap = atoll(e);
    const epic_status sc = note_capture(t, st);
    if (sc != EPIC_OK) return sc;
    t->last = st;
    t->n_vkernels += 1;
    t->nk = 1;
    t->kname[0] = "k_validate_cta";
    mark(t, 0, st);
    launch_validate_cta((int)std::min<long long>(total, t->ctas), st, t->dgl, t->d_table, t->vocab, d_x, n, d_pos, k,
                        d_cand, K, total, d_valid, pack_of(t), cap, 0, t->d_stats);
    mark(t, 1, st);
    return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
  }
  epic_status s = ensure_wworkspace(t, total, n, st);
  if (s == EPIC_OK) s = note_capture(t, st);
  if (s != EPIC_OK) return s;
  t->last = st;
  cudaMemsetAsync(t->d_counter, 0, 8, st);
  // spread the walks over every SM: no more warps per CTA than walks per SM
  const int per_sm = (t->wwarps + sm_count() - 1) / sm_count();
  const int wpc = std::max(1, std::min(kWarpsPerCta, per_sm));
  t->n_vkernels += 1;
  t->nk = 1;
  t->kname[0] = "k_validate_warp";
  mark(t, 0, st);
  launch_validate_warp(t->wwarps / wpc, 32 * wpc, st, t->dgl, t->d_table, t->vocab, d_x, n, d_pos, k, d_cand, K, total,
                       d_valid, wpack_of(t), 0, t->d_counter, t->d_stats);
  mark(t, 1, st);
  return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

int epic_last_kernel_times(const epic_lexer_table* t, float* ms, const char** names, int cap) {
  if (!t || (!ms && cap > 0) || cap < 0) return -1;
  int n = 0;
  if (t->nk > 0) {
    for (int i = 0; i <= t->nk; ++i)
      if (!t->kev[i]) return -1;
    if (cudaEventSynchronize(t->kev[t->nk]) != cudaSuccess) return -1;
    for (int i = 0; i < t->nk && n < cap; ++i, ++n) {
      if (cudaEventElapsedTime(&ms[n], t->kev[i], t->kev[i + 1]) != cudaSuccess) return -1;
      if (names) names[n] = t->kname[i];
    }
  }
  if (t->sel_timed) {
    static const char* sname[2] = {"k_select_spec", "k_select"};
    if (cudaEventSynchronize(t->sev[2]) != cudaSuccess) return -1;
    for (int i = 0; i < 2 && n < cap; ++i, ++n) {
      if (cudaEventElapsedTime(&ms[n], t->sev[i], t->sev[i + 1]) != cudaSuccess) return -1;
      if (names) names[n] = sname[i];
    }
  }
  return n;
}

}  // extern "C"

// ---------------------------------------------------------------- no-alloc validation
// Scratch of epic_validate_batch_noalloc: a fixed device array that every GPU
// which loads this library holds until the process exits.  Its first 256
// bytes hold the work counter; the rest is carved into per-warp workspaces.
constexpr size_t kNoAllocBytes = (size_t)128 << 20;
constexpr int kNoAllocWideMaxN = 128;  // row length limit when item sets exceed 32 words
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

namespace {
std::mutex g_noalloc_mu;
void* g_noalloc_ptr[256] = {nullptr};  // device address of the array, per device ordinal
}  // namespace

extern "C" {

epic_status epic_validate_batch_noalloc(const epic_grammar* g, const epic_lexer_table* tc, const int32_t* d_x,
                                        int32_t B, int32_t n, const int32_t* d_pos, int32_t k,
                                        const int32_t* d_cand, int32_t K, uint8_t* d_valid, void* cuda_stream) {
  epic_lexer_table* t = const_cast<epic_lexer_table*>(tc);
  if (!g || !t || t->g != g || B < 0 || n < 0 || k < 0 || K < 0) return EPIC_ERR_INVALID_ARG;
  long long total = (long long)B * k * K;
  if (total == 0) return EPIC_OK;
  if (!d_x || !d_pos || !d_cand || !d_valid || n == 0) return EPIC_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return EPIC_ERR_CUDA;
  char* base = nullptr;
  {
    // set-up, once per device, with that device current: host code may not
    // use the array's name as a device address
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return EPIC_ERR_CUDA;
      g_noalloc_ptr[dev] = p;
    }
    base = (char*)g_noalloc_ptr[dev];
  }
  const int W = g->dg.W;
  // Wide item sets walk the whole graph per check with rows in the global
  // stage, which takes seconds per check on long rows of large grammars; the
  // fixed array holds too few walks for that to finish in reasonable time,
  // so such calls are limited to short rows.
  if (W > 32 && n > kNoAllocWideMaxN) return EPIC_ERR_CAPACITY;
  WPack wp;
  wp.base = base + 256;
  wp.nmax = std::min(kWCols, 8 * n + 256);
  wp.emax = 256ll * n;
  wp.W = W;
  wp.per_warp = wbytes_per_warp(wp.nmax, wp.emax, W);
  if (wp.per_warp > kNoAllocBytes - 256) {
    // One walk's workspace does not fit the array.  Rows are padded to four
    // words: when the padding is what does not fit, the walk takes the entries
    // that do (more than three quarters of 256 n: the padding is largest for
    // one-word rows, 20 bytes an entry against 16).
    if (wbytes_unpadded(wp.nmax, wp.emax, (g->dg.D + 31) / 32, g->dg.VW) > kNoAllocBytes - 256) return EPIC_ERR_CAPACITY;
    wp.emax = (long long)((kNoAllocBytes - 1024 - wbytes_per_warp(wp.nmax, 0, W)) / (4 + 4 * (size_t)W));
    wp.per_warp = wbytes_per_warp(wp.nmax, wp.emax, W);
  }
  const long long fit = (long long)((kNoAllocBytes - 256) / wp.per_warp);
  {
    WsPack p;
    p.base = base + 256;
    p.dims.nmax = wp.nmax;
    p.dims.emax = wp.emax;
    p.W = W;
    p.VW = g->dg.VW;
    p.FW = 0;
    p.per_cta = ws_bytes_per_cta(p.dims, W, p.VW, 0);
    const long long ctas = std::min<long long>({total, (long long)((kNoAllocBytes - 256) / p.per_cta),
                                                (long long)sm_count()});
    // The array holds fewer walks than there are SMs, and about as many of
    // either kind (256 n entries each: JSON 4 x 128, 71 or 72), so the warp
    // walks have no more of them running and a CTA walk is the faster one: JSON
    // 256 checks 4 x 128 13 ms against 18, 512 checks in eight rounds 23 against
    // 32.  The rule stops at four rounds, short of where a warp each would win:
    // 4 x 256, 256 checks 43 against 71 ms, 8 x 160, 1,152 checks 69 against
    // 102; rows under 96 tokens are even at four rounds (4 x 64, 512 checks 5.9
    // against 5.7).
    if (ctas >= 1 && (cta_walks(total, n, W, ctas) || (n >= 96 && W > 4 && total <= 4 * ctas))) {
      t->last = st;
      t->n_vkernels += 1;
      launch_validate_cta((int)ctas, st, t->dgl, t->d_table, t->vocab, d_x, n, d_pos, k, d_cand, K, total, d_valid, p,
                          wp.emax, 1, t->d_stats);
      return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
    }
  }
  unsigned long long* counter = (unsigned long long*)base;
  // the kernel reads the table's lex entries and adds into its counters:
  // epic_get_stats and epic_lexer_table_destroy synchronize this stream
  t->last = st;
  if (cudaMemsetAsync(counter, 0, sizeof(unsigned long long), st) != cudaSuccess) return EPIC_ERR_CUDA;
  t->n_vkernels += 1;
  const long long warps = std::min<long long>({total, fit, (long long)sm_count() * 2 * kWarpsPerCta});
  // as many warps per CTA as walks per SM
  const int per_cta = (int)std::max<long long>(
      1, std::min<long long>(kWarpsPerCta, (warps + sm_count() - 1) / sm_count()));
  launch_validate_warp((int)(warps / per_cta), 32 * per_cta, st, t->dgl, t->d_table, t->vocab, d_x, n, d_pos, k, d_cand, K,
                       total, d_valid, wp, 1, counter, t->d_stats);
  return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

epic_status epic_pick_candidates(const int32_t* d_cand, const float* d_cand_conf, const uint8_t* d_valid, int32_t B,
                                 int32_t k, int32_t K, int32_t* d_tok, float* d_conf, void* cuda_stream) {
  if (B < 0 || k < 0 || K < 0) return EPIC_ERR_INVALID_ARG;
  long long total = (long long)B * k;
  if (total == 0) return EPIC_OK;
  if (!d_cand || !d_cand_conf || !d_valid || !d_tok || !d_conf) return EPIC_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  k_pick<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(d_cand, d_cand_conf, d_valid, B, k, K, d_tok, d_conf);
  return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

epic_status epic_select_compatible_subset(const epic_grammar* g, const epic_lexer_table* tc, const int32_t* d_x,
                                          int32_t B, int32_t n, const int32_t* d_pos, int32_t k,
                                          const int32_t* d_tok, const float* d_conf, uint8_t* d_selected,
                                          void* cuda_stream) {
  epic_lexer_table* t = const_cast<epic_lexer_table*>(tc);
  if (!g || !t || t->g != g || B < 0 || n < 0 || k < 0 || k > kMaxSel) return EPIC_ERR_INVALID_ARG;
  if ((long long)B * k == 0) return EPIC_OK;
  if (!d_x || !d_pos || !d_tok || !d_conf || !d_selected || n == 0) return EPIC_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int want = std::min(2 * B, sm_count() * 2);
  epic_status s = ensure_workspace(t, plan_workspace(t, want, n), st);
  if (s != EPIC_OK) return s;
  if (t->spec_cap < B) {
    release(t, &t->d_spec);
    t->spec_cap = 0;
    if (!device_alloc(&t->d_spec, (size_t)2 * B)) return EPIC_ERR_OOM;
    t->spec_cap = B;
  }
  s = note_capture(t, st);
  if (s != EPIC_OK) return s;
  t->last = st;
  mark_event(&t->sev[0], st);
  launch_select_spec(std::min(2 * B, t->ctas), st, t->dgl, t->d_table, t->vocab, d_x, B, n, d_pos, k, d_tok,
                     t->d_spec, pack_of(t));
  mark_event(&t->sev[1], st);
  int ctas = std::min(B, t->ctas);
  launch_select(ctas, st, t->dgl, t->d_table, t->vocab, d_x, B, n, d_pos, k, d_tok, d_conf, d_selected, pack_of(t),
                t->d_spec, t->d_stats);
  mark_event(&t->sev[2], st);
  t->sel_timed = t->sev[0] && t->sev[1] && t->sev[2];
  return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

epic_status epic_fallback_commit(const epic_grammar* g, const epic_lexer_table* tc, int32_t* d_x, int32_t B,
                                 int32_t n, const int32_t* d_pos, int32_t k, const int32_t* d_cand,
                                 const float* d_cand_conf, int32_t K, const int32_t* d_n_target,
                                 const uint8_t* d_selected, const uint8_t* d_valid, int32_t* d_filled,
                                 void* cuda_stream) {
  epic_lexer_table* t = const_cast<epic_lexer_table*>(tc);
  if (!g || !t || t->g != g || B < 0 || n < 0 || k < 0 || K < 0) return EPIC_ERR_INVALID_ARG;
  if ((long long)B * k == 0) return EPIC_OK;
  if ((long long)k * K > kMaxFallbackCand) return EPIC_ERR_CAPACITY;
  if (!d_x || !d_pos || !d_cand || !d_cand_conf || !d_n_target || !d_filled || n == 0 || K == 0)
    return EPIC_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const int nc = k * K;
  // rounds of m tests per sequence, one CTA per SM (at most kMaxFallbackSpec
  // tests per sequence, at least one): tests after a round's first pass are
  // spent, and a walk with an SM to itself has twice the warps.  One against
  // two CTAs per SM (molecules, four commits a row): 24 x 96 32 against 42 ms;
  // 64 tokens, 77 rows 31.4 against 30.6, 96 rows 28.3 against 26.3, 128 rows
  // 28.8 against 31.5, 152 rows 28.8 against 31.3.
  int m = std::max(1, std::min(kMaxFallbackSpec, std::min(nc, sm_count() / B)));
  epic_status s = ensure_workspace(
      t, plan_workspace(t, (int)std::min((long long)B * m, (long long)sm_count() * 2), n), st);
  if (s != EPIC_OK) return s;
  m = std::max(1, std::min(m, t->ctas / B));
  auto r16 = [](size_t b) { return (b + 15) & ~(size_t)15; };
  const size_t o_fb = r16((size_t)B * nc), o_res = o_fb + r16((size_t)B * 2 * 4),
               o_act = o_res + r16((size_t)B * m * 2 * 4), need = o_act + 16;
  s = grow(t, &t->d_fb, &t->fb_bytes, need);
  if (s != EPIC_OK) return s;
  t->last = st;
  uint8_t* rej = (uint8_t*)t->d_fb;
  int32_t* fb = (int32_t*)(t->d_fb + o_fb);
  int32_t* res = (int32_t*)(t->d_fb + o_res);
  unsigned long long* act = (unsigned long long*)(t->d_fb + o_act);
  unsigned long long h_act = 0;
  auto read_active = [&]() -> bool {
    if (cudaMemcpyAsync(&h_act, act, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess) return false;
    return cudaStreamSynchronize(st) == cudaSuccess;
  };
  if (cudaMemsetAsync(act, 0, 8, st) != cudaSuccess) return EPIC_ERR_CUDA;
  launch_fallback_init(B, st, n, d_pos, k, d_cand_conf, K, d_n_target, d_selected, d_valid, d_filled, rej, fb, act,
                       t->d_stats);
  if (!read_active()) return EPIC_ERR_CUDA;
  const int grid = (int)std::min<long long>((long long)B * m, t->ctas);
  for (int round = 0; round <= nc && h_act > 0; ++round) {  // each round rejects or commits a candidate
    launch_fallback_round(grid, st, t->dgl, t->d_table, t->vocab, d_x, B, n, d_pos, k, d_cand, d_cand_conf, K, m, rej,
                          fb, res, pack_of(t), t->d_stats);
    if (cudaMemsetAsync(act, 0, 8, st) != cudaSuccess) return EPIC_ERR_CUDA;
    launch_fallback_resolve(B, st, d_x, n, d_pos, k, d_cand, K, m, rej, fb, res, d_filled, act, t->d_stats);
    ++t->n_fb_rounds;
    if (!read_active()) return EPIC_ERR_CUDA;
  }
  return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

epic_status epic_extract_witness(const epic_grammar* g, const epic_lexer_table* tc, const int32_t* d_x, int32_t B,
                                 int32_t n, int32_t* d_terms, int32_t cap, int32_t* d_len, void* cuda_stream) {
  epic_lexer_table* t = const_cast<epic_lexer_table*>(tc);
  if (!g || !t || t->g != g || B < 0 || n < 0 || cap < 1) return EPIC_ERR_INVALID_ARG;
  if (B == 0) return EPIC_OK;
  if (!d_x || !d_terms || !d_len || n == 0) return EPIC_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  SeqPack sp;
  epic_status s = region_prepare(g, t, d_x, B, n, sp, st);
  if (s != EPIC_OK) return s;
  const size_t per = witness_scratch_bytes(cap, t->dgl.D, t->dgl.W, t->dgl.VW);
  s = grow(t, &t->d_wit, &t->wit_bytes, per * (size_t)B);
  if (s == EPIC_OK) s = note_capture(t, st);
  if (s != EPIC_OK) return s;
  launch_witness(B, st, t->dgl, sp, d_terms, cap, d_len, t->d_wit, t->d_stats);
  return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

epic_status epic_commit(int32_t* d_x, int32_t B, int32_t n, const int32_t* d_pos, int32_t k, const int32_t* d_tok,
                        const uint8_t* d_selected, void* cuda_stream) {
  if (B < 0 || n < 0 || k < 0) return EPIC_ERR_INVALID_ARG;
  long long total = (long long)B * k;
  if (total == 0) return EPIC_OK;
  if (!d_x || !d_pos || !d_tok || !d_selected) return EPIC_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  k_commit<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(d_x, B, n, d_pos, k, d_tok, d_selected);
  return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

epic_status epic_get_stats(const epic_lexer_table* t, epic_stats* out, size_t out_bytes, int reset) {
  if (!t || !out || out_bytes < sizeof(epic_stats)) return EPIC_ERR_INVALID_ARG;
  unsigned long long h[S_N];
  if (cudaStreamSynchronize(t->last) != cudaSuccess) return EPIC_ERR_CUDA;
  if (cudaMemcpy(h, t->d_stats, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return EPIC_ERR_CUDA;
  out->checks = h[S_CHECKS];
  out->valid = h[S_VALID];
  out->overflow = h[S_OVERFLOW];
  out->bad_inputs = h[S_BAD];
  out->columns = h[S_COLUMNS];
  out->entries = h[S_ENTRIES];
  out->cover_checks = h[S_COVER];
  out->exact_checks = h[S_EXACT];
  out->selected = h[S_SELECTED];
  out->lex_lookups = h[S_LEX_LOOKUPS];
  out->lex_misses = h[S_LEX_MISSES];
  out->lex_uncached = h[S_LEX_UNCACHED];
  out->witness_failures = h[S_WITNESS_FAIL];
  out->fallback_rounds = t->n_fb_rounds;
  out->fallback_checks = h[S_FB_CHECKS];
  out->fallback_commits = h[S_FB_COMMITS];
  out->region_checks = t->n_region;
  out->validate_kernels = t->n_vkernels;
  if (reset) {
    if (cudaMemset(t->d_stats, 0, sizeof(h)) != cudaSuccess) return EPIC_ERR_CUDA;
    t->n_region = 0;
    t->n_vkernels = 0;
    t->n_fb_rounds = 0;
  }
  return EPIC_OK;
}

}  // extern "C"
