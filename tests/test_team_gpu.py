"""The ordered-list phases of a round (the selection's ordering, the rebalancing
sub-rounds, the move sequence, the best prefix) as one cooperative launch each: traces equal to the
oracle's where the launch changes shape.  Up to 8192 nodes one CTA runs a
phase; beyond, the lists are cut into warp segments over several CTAs.  Block
counts beyond 256 need several sort passes (and a rebalancing sub-round sorts
by block), scores and blocks of more than 32 bits together a wider sort item,
heavy nodes 128-bit rebalancing keys."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from tests.test_parity_gpu import _compare_traces

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def upr():
    from paper_2308_15494_gb300 import build
    build.build()
    import paper_2308_15494_gb300 as m
    m.load()
    return m


CASES = {
    "one_cta_full": lambda: synth.random_small(61, 8192, 6.0, 7, hubs=1),
    "two_ctas_edge": lambda: synth.random_small(62, 8193, 6.0, 2, weighted=False),
    "many_ctas_ragged": lambda: synth.random_small(63, 30011, 5.0, 16, isolated=5),
    "blocks_two_passes": lambda: synth.random_small(64, 12001, 6.0, 300, weighted=False),
    "wide_items": lambda: synth.random_small(65, 9001, 6.0, 11, max_ew=1 << 26),
    "wide_items_one_cta": lambda: synth.random_small(66, 700, 6.0, 8, max_ew=1 << 26),
    "blocks_sorted_weighted": lambda: synth.random_small(68, 12001, 6.0, 300),
    "wide_rebalancing_keys": lambda: synth.random_small(69, 9001, 6.0, 8, max_vw=(1 << 24) - 1, max_ew=1 << 20),
    "heavy_nodes": lambda: synth.random_small(67, 20000, 4.0, 5, max_vw=1000),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_round_traces(upr, name):
    w = CASES[name]()
    ctx = upr.create_from_workload(w)
    part = w.part
    for r in (1, 3):
        rc, p, t = upr.upr_debug_round(ctx, part, r, 4)
        rc0, p0, _, o = oracle.run_round(w, part, r, 4)
        assert rc == rc0
        _compare_traces(t, o)
        assert np.array_equal(p, p0)


@pytest.mark.parametrize("n", [3000, 15001])
def test_repair_of_an_imbalanced_input(upr, n):
    w = synth.random_small(71, n, 5.0, 6, balanced=False)
    ctx = upr.create_from_workload(w)
    rc, p, t = upr.upr_debug_round(ctx, w.part, 0, 4, rebalance_only=True)
    rc0, p0, _, o = oracle.run_round(w, w.part, 0, 4, rebalance_only=True)
    assert rc == rc0
    _compare_traces(t, o)
    assert np.array_equal(p, p0)


def test_appended_sequence_and_guard_over_several_ctas(upr):
    w = synth.random_small(72, 12000, 6.0, 9)
    for over in ({"append": 1}, {"lock_rebalanced": 1}):
        prm = upr.upr_params_default()
        for key, val in over.items():
            setattr(prm, key, val)
        p = w.part.copy()
        st = upr.upr_refine(upr.create_from_workload(w, params=prm), p, 3)
        rc0, p0, c0, _ = oracle.refine(w, w.part, rounds=3, p=oracle.params(**over))
        assert rc0 == oracle.OK and np.array_equal(p, p0) and st.cut_out == c0


@pytest.mark.parametrize("count,k", [(3, 5), (40, 12)])
def test_batch_over_several_ctas(upr, count, k):
    ws = [synth.random_small(80 + i, 700 + 37 * i, 5.0, k, balanced=i % 5 != 4) for i in range(count)]
    ctx = upr.create_batch_from_workloads(ws)
    part = np.concatenate([w.part for w in ws]).astype(np.int32)
    status, _, cut, _ = upr.upr_batch_refine(ctx, part, 3)
    for i, w in enumerate(ws):
        rc0, p0, c0, _ = oracle.refine(w, w.part, rounds=3)
        a, b = ctx.offsets[i], ctx.offsets[i + 1]
        if rc0 == oracle.OK:
            assert status[i] == 0 and np.array_equal(part[a:b], p0) and cut[i] == c0, i
        else:
            assert status[i] == upr.UPR_ERR_INFEASIBLE and np.array_equal(part[a:b], w.part), i


@pytest.mark.parametrize("n,deg,k", [(2000, 9.0, 3), (40000, 1.2, 5), (9000, 40.0, 64)])
def test_cut_and_block_weights_over_chunks(upr, n, deg, k):
    """Chunks of 8192 entries: several rows each, more rows than are staged
    (many short and empty ones), and rows that span chunks; block weights of
    nodes in block order and not."""
    import torch
    w = synth.random_small(90 + k, n, deg, k, hubs=1 if deg > 9 else 0, isolated=n // 3 if deg < 2 else 0)
    ctx = upr.create_from_workload(w)
    dev = [None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
           for a in (w.xadj, w.adj, w.vwgt, w.adjw)]
    for part in (w.part, np.sort(w.part), np.zeros(n, np.int32)):
        part = np.ascontiguousarray(part, np.int32)
        c0, bw0 = oracle.cut(w, part)
        c, bw = upr.upr_cut(ctx, part)
        assert c == c0 and np.array_equal(bw, bw0)
        c, bw = upr.upr_cut_noalloc(dev[0], dev[1], torch.from_numpy(part).cuda(), k, vwgt=dev[2], adjw=dev[3])
        assert c == c0 and np.array_equal(bw, bw0)
