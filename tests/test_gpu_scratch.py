"""Validation of narrow grammars when the workspaces of its faster ways cannot
be had: a warp walks each check, as long as that fits, with the oracle's bits.
Which way a call took is read from the names of its kernels."""
import os

import numpy as np
import pytest

import oracle
from synth import make_workload

pytestmark = pytest.mark.gpu
NTHREADS = os.cpu_count() or 1

FEW = dict(batch=2, k=4, K=16, n=64)       # 128 checks: a CTA each
REGION = dict(batch=4, k=6, K=16, n=136)   # 384 checks of long rows: by region


def validate(w, dev):
    import torch
    import paper_2606_00722_gb300 as epic
    g = epic.Grammar(w.grammar)
    t = epic.LexTable(g, w.vocab)
    valid = torch.full(w.cand.shape, 9, dtype=torch.uint8, device=dev)
    epic.validate_batch(g, t, *[torch.from_numpy(a).to(dev) for a in (w.x, w.pos, w.cand)], valid)
    return valid.cpu().numpy(), list(t.kernel_times()), t.stats()


@pytest.mark.parametrize('shape,env,route', [
    (FEW, {}, ['k_validate_cta']),
    (FEW, dict(EPIC_WORKSPACE_MB='1'), ['k_validate_warp']),         # not one chart fits
    (FEW, dict(EPIC_WORKSPACE_MB='64'), ['k_validate_warp']),        # some do, not one per check
    (FEW, dict(EPIC_ENTRIES_PER_CTA='500'), ['k_validate_warp']),    # charts smaller than a warp's
    (FEW, dict(EPIC_WORKSPACE_MB='1000000000', EPIC_ENTRIES_PER_CTA='10000000000'), ['k_validate_warp']),
    (REGION, {}, ['k_forward_gs', 'k_good', 'k_check']),
    (REGION, dict(EPIC_SEQ_WORKSPACE_MB='1000000000', EPIC_SEQ_ENTRIES='100000000000'), ['k_validate_warp']),
])
def test_narrow_grammars_answer_without_the_faster_workspaces(cuda, monkeypatch, shape, env, route):
    """A small budget, or (the sizes no GPU has) an allocation that fails."""
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    w = make_workload('json-schema', 48, **shape)
    got, kernels, st = validate(w, cuda)
    assert kernels == route and st['overflow'] == 0
    ref = oracle.Oracle(w.grammar, w.vocab).validate_batch(w.x, w.pos, w.cand, nthreads=NTHREADS)
    np.testing.assert_array_equal(got, ref)


def test_a_failed_allocation_leaves_later_calls_alone(cuda, monkeypatch):
    """Forced by region without memory for the charts: out of memory, and the
    same table answers the next call."""
    import torch
    import paper_2606_00722_gb300 as epic
    w = make_workload('json-schema', 49, **FEW)
    g = epic.Grammar(w.grammar)
    t = epic.LexTable(g, w.vocab)
    dev = [torch.from_numpy(a).to(cuda) for a in (w.x, w.pos, w.cand)]
    valid = torch.full(w.cand.shape, 9, dtype=torch.uint8, device=cuda)
    with monkeypatch.context() as m:
        for k, v in dict(EPIC_REGION='1', EPIC_SEQ_WORKSPACE_MB='1000000000', EPIC_SEQ_ENTRIES='100000000000').items():
            m.setenv(k, v)
        with pytest.raises(epic.EpicError) as e:
            epic.validate_batch(g, t, *dev, valid)
        assert e.value.status == 4  # EPIC_ERR_OOM
    epic.validate_batch(g, t, *dev, valid)
    ref = oracle.Oracle(w.grammar, w.vocab).validate_batch(w.x, w.pos, w.cand, nthreads=NTHREADS)
    np.testing.assert_array_equal(valid.cpu().numpy(), ref)


@pytest.mark.parametrize('shape,kernels', [(dict(batch=1, k=2, K=8, n=64), ['k_validate_cta']),
                                           (dict(batch=2, k=9, K=9, n=64), ['k_validate_warp']),
                                           (dict(batch=2, k=10, K=16, n=136), ['k_forward_gs', 'k_good', 'k_check'])])
def test_captured_validation_outlives_larger_calls(cuda, shape, kernels):
    """A graph of validation keeps its workspace when later calls on the same
    table (larger selections, witnesses and validations) need more: replays
    on new rows still equal the oracle."""
    import torch
    import paper_2606_00722_gb300 as epic
    w = make_workload('json-schema', 50, **shape)
    more = make_workload('json-schema', 50, **dict(shape, batch=2 * w.B))  # the same vocabulary
    rows = [(w.x, w.pos, w.cand), (more.x[w.B:], more.pos[w.B:], more.cand[w.B:])]
    assert more.vocab == w.vocab and not np.array_equal(rows[0][0], rows[1][0])
    big = make_workload('json-schema', 50, batch=40, k=4, K=16, n=shape['n'] + 8)
    g = epic.Grammar(w.grammar)
    t = epic.LexTable(g, w.vocab)
    put = lambda *a: [torch.from_numpy(v).to(cuda) for v in a]
    x, pos, cand = put(w.x, w.pos, w.cand)
    valid = torch.full(w.cand.shape, 9, dtype=torch.uint8, device=cuda)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        epic.validate_batch(g, t, x, pos, cand, valid)
    side.synchronize()
    assert list(t.kernel_times()) == kernels
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        epic.validate_batch(g, t, x, pos, cand, valid)
    # every workspace grows
    bx, bpos, bcand, btok, bconf = put(big.x, big.pos, big.cand, big.cand[:, :, 0].copy(), big.conf[:, :, 0].copy())
    bvalid = torch.empty(big.cand.shape, dtype=torch.uint8, device=cuda)
    sel = torch.empty(big.pos.shape, dtype=torch.uint8, device=cuda)
    lens = torch.empty(40, dtype=torch.int32, device=cuda)
    for _ in range(2):
        epic.validate_batch(g, t, bx, bpos, bcand, bvalid)
        epic.select_compatible_subset(g, t, bx, bpos, btok, bconf, sel)
        epic.extract_witness(g, t, bx, torch.zeros((40, 8 * big.n), dtype=torch.int32, device=cuda), lens)
    fill = torch.full((1 << 28,), 255, dtype=torch.uint8, device=cuda)  # whatever was given back is someone else's now
    O = oracle.Oracle(w.grammar, w.vocab)
    for arrays in rows + rows[:1]:
        for d, a in zip((x, pos, cand), arrays):
            d.copy_(torch.from_numpy(a))
        valid.fill_(9)
        graph.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(valid.cpu().numpy(), O.validate_batch(*arrays, nthreads=NTHREADS))
    del fill, graph
