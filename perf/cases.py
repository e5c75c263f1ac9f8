"""Performance cases of the constraint work of one denoising step.

A case is one call (or one whole step) that a decoding program makes on a
batch of partial outputs: a grammar of ``synth/`` with its vocabulary, a batch
of rows, k proposed positions per row and K candidate tokens per position.
Every case goes through the package's public functions on device tensors, as
a serving loop would call them.

What a program keeps from step to step -- the compiled grammar and the lexing
table -- is made once per grammar and vocabulary and shared by the states of
one case; the rows, masks, proposals and candidates come from the seed.

Outputs are validity bits, token ids and selection marks (and the picked
candidates' own confidences, copied): whole values with one right answer, so
they are compared exactly, and there is no 64-bit value to set beside them.
"""
import math

import numpy as np
import torch

import paper_2606_00722_gb300 as epic
from synth.grammars import grammar_for
from synth.workload import WORKLOADS, _sentence_tokens, make_vocab, render, sample_derivation

# Lexer states of each grammar: a token inside a span is looked up from every state that is live there, all of them
# right after a gap.
_STATES = {'expr-tiny': 11, 'json-schema': 183, 'clike-512': 209, 'random-stress-1024': 307, 'smiles-256': 49}


def _case(name, op, grammar, batch, n, k, K, lazy=0, mask=None):
    return {'name': name, 'op': op, 'grammar': grammar, 'batch': batch, 'n': n, 'k': k, 'K': K, 'lazy': lazy,
            'mask': WORKLOADS[grammar].mask_rate if mask is None else mask}


def listed():
    return [
        # the smallest decoding step there is: one short row, where launches, host round trips and the latency of a
        # few tens of columns are all of the time
        _case('expr-step', 'step', 'expr-tiny', 1, 32, 8, 8),
        # a serving process whose memory belongs to its own pool checks a few short rows without allocating
        _case('json-noalloc', 'noalloc', 'json-schema', 4, 128, 4, 16),
        # the checks of one step of schema-constrained JSON decoding, at the configuration's own size
        _case('json-validate', 'validate', 'json-schema', 16, 256, 4, 16),
        # a whole step with the lexing memo filled on use, late in decoding (few masks left), odd sizes
        _case('json-step-lazy', 'step', 'json-schema', 11, 173, 5, 13, lazy=1 << 20, mask=0.3),
        # recovery from a failure: one completion of every row of the batch
        _case('json-witness', 'witness', 'json-schema', 16, 256, 4, 16),
        # the largest batch: molecule strings, many short-lexeme rows at once
        _case('smiles-validate', 'validate', 'smiles-256', 256, 256, 4, 16),
        # choosing the parallel commit among many proposed positions, odd sizes
        _case('smiles-select', 'select', 'smiles-256', 48, 144, 16, 16),
        # no parallel batch survived: commits one after another by the rejection loop
        _case('smiles-fallback', 'fallback', 'smiles-256', 24, 96, 4, 16),
        # code under a grammar of hundreds of productions: a few short rows (an interactive completion) ...
        _case('code-validate-small', 'validate', 'clike-512', 8, 96, 8, 32),
        # ... a full batch of longer ones ...
        _case('code-validate', 'validate', 'clike-512', 32, 256, 8, 32),
        # ... and a whole step early in decoding (most positions masked), odd sizes
        _case('code-step', 'step', 'clike-512', 3, 151, 7, 32, mask=0.7),
        # the widest grammar (400 nonterminals, 1,500 productions) on rows that one call answers quickly
        _case('wide-validate', 'validate', 'random-stress-1024', 4, 96, 8, 16),
    ]


# (op, grammar, rows, row length, proposals, candidates): the ranges that the listed cases stand for; a range that spans
# more than a factor of ten is drawn over its logarithm
_RANGES = [
    ('step', 'expr-tiny', (1, 16), (8, 48), (1, 8), (2, 16)),
    ('validate', 'expr-tiny', (1, 64), (8, 48), (1, 8), (2, 16)),
    ('noalloc', 'json-schema', (1, 8), (24, 160), (1, 6), (4, 24)),
    ('validate', 'json-schema', (1, 24), (24, 256), (1, 16), (4, 32)),
    ('step', 'json-schema', (1, 16), (24, 224), (2, 8), (4, 24)),
    ('witness', 'json-schema', (1, 24), (24, 256), (2, 4), (4, 16)),
    ('validate', 'smiles-256', (2, 256), (24, 224), (1, 8), (4, 24)),
    ('select', 'smiles-256', (1, 64), (32, 144), (2, 20), (4, 16)),
    ('fallback', 'smiles-256', (1, 32), (24, 104), (1, 5), (4, 24)),
    ('validate', 'clike-512', (1, 32), (24, 200), (1, 10), (8, 48)),
    ('step', 'clike-512', (1, 6), (24, 144), (2, 8), (8, 40)),
    ('witness', 'clike-512', (1, 16), (24, 160), (2, 4), (4, 16)),
    ('validate', 'random-stress-1024', (1, 8), (16, 96), (1, 10), (4, 24)),
]


def draw(rng):
    op, grammar, *ranges = rng.choice(_RANGES)
    v = [round(math.exp(rng.uniform(math.log(lo), math.log(hi)))) if hi > 10 * lo else rng.randint(lo, hi)
         for lo, hi in ranges]
    v[2] = min(v[2], max(1, v[1] // 4))
    lazy = rng.choice([0, 0, 0, 1 << 20, 1 << 14])
    c = _case('', op, grammar, *v, lazy=lazy, mask=round(rng.uniform(0.25, 0.75), 2))
    del c['name']
    return c


def work(case):
    """Bytes that one pass cannot do without: every input and output once, and the lexing-table entries of the fixed
    tokens' and candidates' first lookups (every lexer state, 16 bytes each).  The recognition itself is bit operations
    on sets whose number depends on the text; it is not counted."""
    B, n, k, K, op = case['batch'], case['n'], case['k'], case['K'], case['op']
    row = 16 * _STATES[case['grammar']]
    fixed = int(B * n * (1 - case['mask']))
    b = 4 * B * n + fixed * row
    if op != 'witness':
        b += 4 * B * k + (4 * B * k * K if op != 'select' else 8 * B * k)
    if op in ('validate', 'noalloc', 'step'):
        b += B * k * K * (5 + row) + 8 * B * k
    if op == 'select':
        b += 4 * B * n + B * k
    if op in ('step', 'fallback'):
        b += 4 * B * n + 4 * B * k * K + 9 * B * k
    if op == 'witness':
        b += 4 * B * (4 * n + 1)
    return {'bytes': float(b), 'flops': 0.0}


# ---------------------------------------------------------------- inputs

_vocab_memo = {}   # grammar name -> (grammar, vocabulary, sentence pools)
_handle = {}       # the one compiled grammar and lexing table in use: {key: (Grammar, LexTable)}


def _language(name):
    """The grammar, its vocabulary (both the same for every seed) and a dict of sentence pools by row length."""
    if name not in _vocab_memo:
        g = grammar_for(name)
        rng = np.random.Generator(np.random.PCG64(7))
        samples = [render(g, sample_derivation(g, rng, 40), rng) for _ in range(64)]
        vocab = make_vocab(g, WORKLOADS[name], rng, samples)
        _vocab_memo[name] = (g, vocab, {})
    return _vocab_memo[name]


def _sentences(name, n, count):
    """A pool of token sentences of at most n tokens (the same for every seed; a row is one of them under its own mask)."""
    g, vocab, pools = _language(name)
    pool = pools.setdefault(n, [])
    if len(pool) < count:
        rng = np.random.Generator(np.random.PCG64(1000003 + n))
        index = {t: i for i, t in enumerate(vocab)}
        maxlen = max(len(t) for t in vocab)
        pool[:] = [np.array(_sentence_tokens(g, rng, index, maxlen, n), np.int32) for _ in range(count)]
    return pool


def _compiled(case):
    """The compiled grammar and lexing table of the case (kept while cases of the same key run)."""
    key = (case['grammar'], case['lazy'], case['op'], case['n'])
    if key not in _handle:
        _handle.clear()
        g, vocab, _ = _language(case['grammar'])
        G = epic.Grammar(g)
        t = epic.LexTable(G, vocab, lazy_capacity=case['lazy'] or None)
        _handle[key] = (G, t)
    return _handle[key]


def prepare(case, seed):
    dev = torch.device('cuda')
    B, n, k, K = case['batch'], case['n'], case['k'], case['K']
    _, vocab, _ = _language(case['grammar'])
    V = len(vocab)
    pool = _sentences(case['grammar'], n, min(48, max(8, B)))
    rng = np.random.Generator(np.random.PCG64(seed))
    x = np.full((B, n), -1, np.int32)
    wit = np.full((B, n), -1, np.int32)
    pos = np.zeros((B, k), np.int32)
    order = rng.permutation(len(pool))
    for b in range(B):
        toks = pool[int(order[b % len(pool)])]
        m = len(toks)
        wit[b, :m] = toks
        x[b, :m] = toks
        extra = max(0, max(k, int(round(case['mask'] * n))) - (n - m))
        if extra > 0:
            x[b, rng.choice(m, size=min(extra, m), replace=False)] = -1
        pos[b] = np.sort(rng.choice(np.flatnonzero(x[b] < 0), size=k, replace=False))
    # K distinct candidates per position: Gumbel-top-K over N(0, 1) logits, the sentence's own token raised so that it
    # is usually among them; confidence = softmax probability
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    own = torch.from_numpy(np.take_along_axis(wit, pos, 1).astype(np.int64).reshape(-1)).to(dev)
    cand = torch.empty((B * k, K), dtype=torch.int32, device=dev)
    conf = torch.empty((B * k, K), dtype=torch.float32, device=dev)
    for lo in range(0, B * k, 512):
        hi = min(B * k, lo + 512)
        logits = torch.randn((hi - lo, V), generator=gen, device=dev)
        o = own[lo:hi]
        row = torch.nonzero(o >= 0).reshape(-1)
        logits[row, o[row]] += math.log(V) + 1.0
        u = torch.rand((hi - lo, V), generator=gen, device=dev).clamp_(1e-12, 1.0 - 1e-7)
        top = torch.topk(logits - torch.log(-torch.log(u)), K, dim=1).indices
        cand[lo:hi] = top.to(torch.int32)
        conf[lo:hi] = torch.gather(torch.softmax(logits, 1), 1, top)
    s = {'case': case, 'x': torch.from_numpy(x).to(dev), 'pos': torch.from_numpy(pos).to(dev),
         'cand': cand.view(B, k, K), 'conf3': conf.view(B, k, K),
         'n_target': torch.full((B,), k, dtype=torch.int32, device=dev)}
    s['bufs'] = dict(valid=torch.empty((B, k, K), dtype=torch.uint8, device=dev),
                     tok=torch.empty((B, k), dtype=torch.int32, device=dev),
                     conf=torch.empty((B, k), dtype=torch.float32, device=dev),
                     selected=torch.empty((B, k), dtype=torch.uint8, device=dev),
                     filled=torch.empty((B, k), dtype=torch.int32, device=dev))
    s['g'], s['t'] = _compiled(case)
    if case['op'] == 'witness':
        s['terms'] = torch.zeros((B, 4 * n), dtype=torch.int32, device=dev)
        s['lens'] = torch.empty((B,), dtype=torch.int32, device=dev)
    if case['op'] in ('select', 'fallback'):
        b = s['bufs']
        epic.validate_batch(s['g'], s['t'], s['x'], s['pos'], s['cand'], b['valid'])
        epic.pick_candidates(s['cand'], s['conf3'], b['valid'], b['tok'], b['conf'])
    return s


def run(s):
    op, b = s['case']['op'], s['bufs']
    if op in ('validate', 'noalloc'):  # the checks, then the best valid candidate of every position
        check = epic.validate_batch if op == 'validate' else epic.validate_batch_noalloc
        check(s['g'], s['t'], s['x'], s['pos'], s['cand'], b['valid'])
        epic.pick_candidates(s['cand'], s['conf3'], b['valid'], b['tok'], b['conf'])
        return [b['valid'], b['tok'], b['conf']]
    if op == 'select':  # choose the parallel commit and make it
        x = s['x'].clone()
        epic.select_compatible_subset(s['g'], s['t'], x, s['pos'], b['tok'], b['conf'], b['selected'])
        epic.commit(x, s['pos'], b['tok'], b['selected'])
        return [x, b['selected']]
    if op == 'fallback':
        x = s['x'].clone()
        epic.fallback_commit(s['g'], s['t'], x, s['pos'], s['cand'], s['conf3'], s['n_target'], None, b['filled'],
                             valid=b['valid'])
        return [x, b['filled']]
    if op == 'witness':
        epic.extract_witness(s['g'], s['t'], s['x'], s['terms'], s['lens'])
        return [s['lens'], s['terms']]
    x = s['x'].clone()
    epic.decode_step(s['g'], s['t'], x, s['pos'], s['cand'], s['conf3'], s['n_target'], b)
    return [x, b['valid'], b['tok'], b['conf'], b['selected'], b['filled']]


def tolerance(case):
    return 'exact'
