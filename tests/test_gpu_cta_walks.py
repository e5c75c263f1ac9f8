"""Whole-graph walks with a CTA per check: small batches on both sides of each
line of the rule that picks them (the kernels' names say which side; 152 SMs),
with and without allocation, against the oracle; a check that runs out of
chart entries reports 2."""
import os

import numpy as np
import pytest

import oracle
from synth import make_workload

from test_gpu_scratch import validate

pytestmark = pytest.mark.gpu
NTHREADS = os.cpu_count() or 1


CTA, WARP, REGION = ['k_validate_cta'], ['k_validate_warp'], ['k_forward_gs', 'k_good', 'k_check']


@pytest.mark.parametrize('name,kw,kernels', [
    ('json-schema', dict(batch=1, n=40, k=1, K=1), CTA),
    ('json-schema', dict(batch=2, n=48, k=9, K=8), CTA),        # one round of walks
    ('json-schema', dict(batch=2, n=48, k=9, K=9), WARP),       # a warp each
    ('json-schema', dict(batch=3, n=97, k=10, K=10), CTA),      # two rounds
    ('json-schema', dict(batch=3, n=97, k=10, K=11), WARP),     # more than two rounds
    ('json-schema', dict(batch=2, n=140, k=10, K=16), REGION),  # the same of a long row
    ('smiles-256', dict(batch=2, n=60, k=5, K=11), CTA),
    ('clike-512', dict(batch=1, n=40, k=4, K=9), REGION),       # wide item sets
    ('expr-tiny', dict(), WARP),                                # tiny ones
    ('expr-tiny', dict(n=131, k=5, K=5), REGION),
])
def test_small_batches(cuda, name, kw, kernels):
    import torch
    import paper_2606_00722_gb300 as epic
    w = make_workload(name, 21, **kw)
    ref = oracle.Oracle(w.grammar, w.vocab).validate_batch(w.x, w.pos, w.cand, nthreads=NTHREADS)
    got, took, st = validate(w, cuda)
    assert took == kernels and st['overflow'] == 0
    np.testing.assert_array_equal(got, ref)
    g = epic.Grammar(w.grammar)
    t = epic.LexTable(g, w.vocab)
    dev = [torch.from_numpy(a).to(cuda) for a in (w.x, w.pos, w.cand)]
    valid = torch.full(w.cand.shape, 9, dtype=torch.uint8, device=cuda)
    for _ in range(2):  # the second call meets the first one's contents of the scratch array
        epic.validate_batch_noalloc(g, t, *dev, valid)
        np.testing.assert_array_equal(valid.cpu().numpy(), ref)


def test_capacity_reports_two(cuda, monkeypatch):
    monkeypatch.setenv('EPIC_ENTRIES_PER_WALK', '60')
    w = make_workload('json-schema', 22, batch=2, k=4, K=6, n=64)
    got, took, st = validate(w, cuda)
    assert took == CTA
    ref = oracle.Oracle(w.grammar, w.vocab).validate_batch(w.x, w.pos, w.cand, nthreads=NTHREADS)
    ovf = got == 2
    assert ovf.any() and st['overflow'] == int(ovf.sum())
    np.testing.assert_array_equal(got[~ovf], ref[~ovf])
