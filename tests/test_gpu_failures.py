"""Failure paths on the GPU, in the safe form: every device loop is bounded,
and a check or a sequence that runs out of a capacity gives up inside its
bounds and reports (value 2 in d_valid, stats.overflow), never faulting or
hanging.  The capacities are made tiny through the library's workspace knobs
so that the limits are reached on ordinary inputs."""
import os

import numpy as np
import pytest

import oracle
from synth import make_workload

from test_gpu_edges import run_gpu
from test_gpu_scratch import validate

pytestmark = pytest.mark.gpu
NTHREADS = os.cpu_count() or 1


@pytest.mark.parametrize('k,K,kernel', [(3, 6, 'k_validate_cta'), (9, 18, 'k_validate_warp')])
def test_whole_walk_overflow_reports_two(cuda, monkeypatch, k, K, kernel):
    """Whole-graph walks, a CTA or a warp per check, with room for 40 chart
    entries: checks whose chart needs more report 2 and are counted; every
    other bit equals the oracle."""
    monkeypatch.setenv('EPIC_REGION', '0')
    monkeypatch.setenv('EPIC_ENTRIES_PER_WALK', '40')
    w = make_workload('json-schema', 42, batch=2, k=k, K=K, n=64)
    got, kernels, st = validate(w, cuda)
    assert kernels == [kernel]
    ref = oracle.Oracle(w.grammar, w.vocab).validate_batch(w.x, w.pos, w.cand, nthreads=NTHREADS)
    ovf = got == 2
    assert ovf.any(), 'the tiny workspace should overflow some checks'
    assert st['overflow'] == int(ovf.sum())
    np.testing.assert_array_equal(got[~ovf], ref[~ovf])
    assert set(np.unique(got)) <= {0, 1, 2}


def test_region_chart_overflow_falls_back_to_whole_walks(cuda, monkeypatch):
    """Per-sequence forward charts with room for 300 entries: sequences whose
    chart does not fit walk their checks whole instead, with the same bits
    as the oracle (nothing is reported as overflow: the whole walks have
    their own room)."""
    monkeypatch.setenv('EPIC_REGION', '1')
    monkeypatch.setenv('EPIC_SEQ_ENTRIES', '300')
    w = make_workload('json-schema', 43, batch=3, k=3, K=5, n=96)
    got, st = run_gpu(w.grammar, w.vocab, w.x, w.pos, w.cand, cuda)
    ref = oracle.Oracle(w.grammar, w.vocab).validate_batch(w.x, w.pos, w.cand, nthreads=NTHREADS)
    assert st['overflow'] == 0
    np.testing.assert_array_equal(got, ref)


def test_both_limits_at_once(cuda, monkeypatch):
    """Forward charts and whole walks both too small: the checks report 2,
    none is silently answered."""
    monkeypatch.setenv('EPIC_REGION', '1')
    monkeypatch.setenv('EPIC_SEQ_ENTRIES', '200')
    monkeypatch.setenv('EPIC_ENTRIES_PER_WALK', '30')
    w = make_workload('json-schema', 44, batch=2, k=2, K=4, n=80)
    got, st = run_gpu(w.grammar, w.vocab, w.x, w.pos, w.cand, cuda)
    ref = oracle.Oracle(w.grammar, w.vocab).validate_batch(w.x, w.pos, w.cand, nthreads=NTHREADS)
    ovf = got == 2
    assert st['overflow'] == int(ovf.sum())
    np.testing.assert_array_equal(got[~ovf], ref[~ovf])
    assert ovf.any()


def bracket_rows(w, rows, free):
    """w's rows, those of `rows` replaced by opening brackets, 13 to a token, with the first and the last `free` tokens
    masked: each token makes a chain of a dozen columns, more than a walk of such a row has room for."""
    vocab = list(w.vocab) + [b'[' * 13]
    x = w.x.copy()
    pos = w.pos.copy()
    n, k = x.shape[1], pos.shape[1]
    for b in rows:
        x[b] = len(vocab) - 1
        x[b, 0] = -1
        x[b, n - free:] = -1
        pos[b] = np.sort(np.resize(np.arange(n - free, n), k))
    return vocab, x, pos


def test_columns_run_out_then_other_checks_in_the_same_cta(cuda):
    """CTA walks that run out of columns (8 n + 256 of them in the
    no-allocation call) in the middle of a token's chain report 2; the checks
    that the same CTAs take before and after them equal the oracle."""
    import torch
    import paper_2606_00722_gb300 as epic
    w = make_workload('json-schema', 45, batch=10, n=100, k=1, K=30)
    long = [1, 4, 5, 7, 8]
    vocab, x, pos = bracket_rows(w, long, 2)
    ref = oracle.Oracle(w.grammar, vocab).validate_batch(x, pos, w.cand, nthreads=NTHREADS)
    g = epic.Grammar(w.grammar)
    t = epic.LexTable(g, vocab)
    dev = [torch.from_numpy(a).to(cuda) for a in (x, pos, w.cand)]
    valid = torch.full(w.cand.shape, 9, dtype=torch.uint8, device=cuda)
    epic.validate_batch_noalloc(g, t, *[a[long].contiguous() for a in dev], valid)
    assert (valid[:len(long)] == 2).all()
    assert t.stats(reset=True)['columns'] == len(long) * w.K * (8 * 100 + 256), 'the columns are what runs out'
    for _ in range(3):
        valid.fill_(9)
        epic.validate_batch_noalloc(g, t, *dev, valid)
        got = valid.cpu().numpy()
        assert (got[long] == 2).all()
        rest = np.delete(np.arange(len(x)), long)
        np.testing.assert_array_equal(got[rest], ref[rest])
    assert t.stats()['overflow'] == 3 * got[long].size
    # by region, the charts that do not fit leave their checks to whole walks with room for 4,096 columns
    epic.validate_batch(g, t, *dev, valid)
    np.testing.assert_array_equal(valid.cpu().numpy(), ref)


def test_columns_run_out_in_selection(cuda, monkeypatch):
    """Selection over fewer CTAs than rows, every other row out of columns
    (4,096): those select nothing and report 2, the others equal the oracle."""
    import torch
    import paper_2606_00722_gb300 as epic
    monkeypatch.setenv('EPIC_WORKSPACE_MB', '64')  # four charts of 400 tokens
    w = make_workload('json-schema', 46, batch=9, n=400, k=4, K=2)
    long = [0, 3, 4, 6, 8]
    vocab, x, pos = bracket_rows(w, long, 4)
    rest = np.delete(np.arange(len(x)), long)
    tok = np.take_along_axis(np.where(w.witness >= 0, w.witness, w.cand[:, 0, :1]), pos, 1).astype(np.int32)
    tok[long] = vocab.index(b']')
    conf = np.random.default_rng(3).random(tok.shape).astype(np.float32)
    g = epic.Grammar(w.grammar)
    t = epic.LexTable(g, vocab)
    sel = torch.full(tok.shape, 9, dtype=torch.uint8, device=cuda)
    epic.select_compatible_subset(g, t, *[torch.from_numpy(a).to(cuda) for a in (x, pos, tok, conf)], sel)
    got = sel.cpu().numpy()
    assert (got[long] == 2).all()
    ref = oracle.Oracle(w.grammar, vocab).select(x[rest], pos[rest], tok[rest], conf[rest])
    assert ref.any()
    np.testing.assert_array_equal(got[rest], ref)
