"""Row shapes and completion chains of the chart walks against the oracle.

A chart row of W item words lies in 4, 16 or 32 lanes depending on W, and the
completions that chain at one origin come from a table that depends on
nullable symbols and on which of the two nodes is a gap.  The grammars here
put W on both sides of every boundary and hold epsilon rules in every place of
a production; every path (whole-graph walks, checks by region, selection, the
rejection fallback) answers small batches bit for bit."""
import dataclasses
import os

import numpy as np
import pytest

import oracle
from synth import grammars as G
from synth.workload import render, sample_derivation, tokenize

from test_gpu_edges import run_gpu

pytestmark = pytest.mark.gpu
NTHREADS = os.cpu_count() or 1


def eps_grammar():
    """Nullable symbols before, after and around the others, unit chains
    through them, and left and right recursion."""
    b = G._Builder('eps-chains')
    b.lit('a', 'A')
    b.lit('b', 'B')
    b.lit('(', 'LP')
    b.lit(')', 'RP')
    b.term('WS', '[ ]+', ('ws',), skip=True)
    b.rule('S', 'N X N', 'X Y', 'S Z')
    b.rule('X', 'Y', 'N Y N', 'LP S RP')
    b.rule('Y', 'Z', 'Z N', 'A X')
    b.rule('Z', 'A', 'N B', 'B N M')
    b.rule('N', '', 'M', 'A N')
    b.rule('M', '', 'N M')
    return b.build('S', 'ab() ')


def padded(spec, extra):
    """The same language with `extra` nonterminals declared ahead of the others that no production uses."""
    T = spec.T
    shift = lambda s: s if s < T else s + extra
    return dataclasses.replace(spec, nonterminals=['unused%d' % i for i in range(extra)] + list(spec.nonterminals),
                               start=spec.start + extra,
                               productions=[(lhs + extra, [shift(s) for s in rhs]) for lhs, rhs in spec.productions])


def item_words(spec):
    items = sum(len(r) + 1 for _, r in spec.productions) + 2
    return (items + 31) // 32


def random_rows(spec, seed, rows, n, k, K):
    """Masked sample sentences (completable) and random rows (mostly not)."""
    rng = np.random.default_rng(seed)
    samples = [render(spec, sample_derivation(spec, rng, max(4, n // 2)), rng).encode('latin-1') for _ in range(rows)]
    vocab = [c.encode('latin-1') for c in sorted(set(spec.charset) | set(''.join(s.decode('latin-1') for s in samples)))]
    vocab += sorted({s[i:i + 3] for s in samples for i in range(0, max(1, len(s) - 3), 2)} - set(vocab))[:60]
    index = {t: i for i, t in enumerate(vocab)}
    x = np.full((rows, n), -1, np.int32)
    for b in range(rows):
        toks = tokenize(samples[b], index, 3)[:n]
        x[b, :len(toks)] = toks
        if b % 3 == 2:
            x[b] = rng.integers(0, len(vocab), n)
        x[b, rng.random(n) < 0.5] = -1
        m = np.flatnonzero(x[b] < 0)
        if len(m) < k:
            x[b, rng.permutation(n)[:k]] = -1
    pos = np.stack([np.sort(rng.choice(np.flatnonzero(x[b] < 0), k, replace=False)) for b in range(rows)]).astype(np.int32)
    cand = rng.integers(0, len(vocab), (rows, k, K)).astype(np.int32)
    conf = rng.random((rows, k, K)).astype(np.float32)
    return vocab, x, pos, cand, conf


GRAMMARS = {'eps': (eps_grammar, None)}
# (nonterminals, productions): item words W at and around 16 and 64
for nt, pr, words in ((30, 95, (13, 16)), (40, 130, (17, 20)), (150, 495, (61, 64)), (160, 515, (65, 68)), (210, 700, (80, 120))):
    GRAMMARS['random-%d-%d' % (nt, pr)] = (
        (lambda nt=nt, pr=pr: G.random_grammar(77 + nt, nt, pr, 40, 5, 0.2, nt % 20 == 0, 'random-%d' % nt)), words)


@pytest.mark.parametrize('name', sorted(GRAMMARS))
@pytest.mark.parametrize('path', ['0', '1'])
def test_rows_against_oracle(cuda, monkeypatch, name, path):
    monkeypatch.setenv('EPIC_REGION', path)
    make, words = GRAMMARS[name]
    spec = make()
    if words:
        assert words[0] <= item_words(spec) <= words[1], item_words(spec)
    n, rows, k, K = (18, 9, 5, 6) if name == 'eps' else (12, 4, 3, 4)
    vocab, x, pos, cand, conf = random_rows(spec, 5, rows, n, k, K)
    got, st = run_gpu(spec, vocab, x, pos, cand, cuda)
    assert st['overflow'] == 0
    O = oracle.Oracle(spec, vocab)
    np.testing.assert_array_equal(got, O.validate_batch(x, pos, cand, nthreads=NTHREADS))


@pytest.mark.parametrize('name,extra,path', [('eps', 160, '1'), ('eps', 1000, '1'), ('eps', 1000, '0'),
                                             ('random-40-130', 980, '1'), ('random-210-700', 800, '1')])
def test_more_declared_nonterminals_than_items(cuda, monkeypatch, name, extra, path):
    """Nonterminals keep their declared numbers and rows hold only the items
    that trimming leaves, so a set of nonterminals can be longer than a row."""
    monkeypatch.setenv('EPIC_REGION', path)
    spec = GRAMMARS[name][0]()
    n, rows, k, K = (18, 9, 5, 6) if name == 'eps' else (12, 4, 3, 4)
    vocab, x, pos, cand, conf = random_rows(spec, 7, rows, n, k, K)
    wide = padded(spec, extra)
    ref = oracle.Oracle(wide, vocab).validate_batch(x, pos, cand, nthreads=NTHREADS)
    np.testing.assert_array_equal(ref, oracle.Oracle(spec, vocab).validate_batch(x, pos, cand, nthreads=NTHREADS))
    got, st = run_gpu(wide, vocab, x, pos, cand, cuda)
    assert st['overflow'] == 0 and ref.any()
    np.testing.assert_array_equal(got, ref)


@pytest.mark.parametrize('name', sorted(GRAMMARS))
def test_step_against_oracle(cuda, name):
    import torch
    import paper_2606_00722_gb300 as epic
    spec = GRAMMARS[name][0]()
    n, rows, k, K = (18, 9, 5, 6) if name == 'eps' else (12, 4, 3, 4)
    vocab, x, pos, cand, conf = random_rows(spec, 6, rows, n, k, K)
    g, t = epic.Grammar(spec), None
    t = epic.LexTable(g, vocab)
    dev = lambda a: torch.from_numpy(a).to(cuda)
    xd = dev(x.copy())
    nt = np.full(rows, k, np.int32)
    bufs = dict(valid=torch.empty(cand.shape, dtype=torch.uint8, device=cuda),
                tok=torch.empty(pos.shape, dtype=torch.int32, device=cuda),
                conf=torch.empty(pos.shape, dtype=torch.float32, device=cuda),
                selected=torch.empty(pos.shape, dtype=torch.uint8, device=cuda),
                filled=torch.empty(pos.shape, dtype=torch.int32, device=cuda))
    epic.decode_step(g, t, xd, dev(pos), dev(cand), dev(conf), dev(nt), bufs)
    torch.cuda.synchronize()
    O = oracle.Oracle(spec, vocab)
    valid = O.validate_batch(x, pos, cand, nthreads=NTHREADS)
    np.testing.assert_array_equal(bufs['valid'].cpu().numpy(), valid)
    tok, cf = oracle.pick_candidates(valid, cand, conf)
    sel = O.select(x, pos, tok, cf)
    np.testing.assert_array_equal(bufs['selected'].cpu().numpy(), sel)
    rx, filled, _ = O.fallback(O.commit(x, pos, tok, sel), pos, cand, conf, nt, sel)
    np.testing.assert_array_equal(bufs['filled'].cpu().numpy(), filled)
    np.testing.assert_array_equal(xd.cpu().numpy(), rx)
