"""All rounds of a call on a small graph in one launch, against the oracle, at
the sizes where its CTAs and their work change: one CTA up to 2048 nodes and
65536 adjacency entries and table cells, eight up to 8192 nodes, sixteen up to
2^19 entries and cells (beyond, step by step); rows of more than 512 entries
(spread over a CTA, at most 256 of them noted) and of more than 4096 (hubs)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def upr():
    from paper_2308_15494_gb300 import build
    build.build()
    import paper_2308_15494_gb300 as m
    m.load()
    return m


def _long_rows_of_one_cta():
    """320 nodes of degree over 512, all of them taken by the first of eight CTAs."""
    rng = np.random.Generator(np.random.PCG64(5))
    n, k = 2560, 3
    ids = np.arange(n)
    a, b = ids[ids % 256 < 32], ids[ids % 256 >= 32]
    src = np.repeat(a, 540)
    dst = np.concatenate([rng.choice(b, 540, replace=False) for _ in a])
    xadj, adj = synth.csr_from_edges(n, src.astype(np.int32), dst.astype(np.int32))
    assert (np.diff(xadj) > 512).sum() == 320
    return synth.Workload("long_rows", n, xadj, adj, None, None, k, 0.03,
                          synth.part_random_balanced(n, k, 6), 3, {})


CASES = {
    "two_nodes": lambda: synth.random_small(101, 2, 4.0, 2, weighted=False),
    "no_edges": lambda: synth.random_small(102, 40, 0.0, 3),
    "one_cta_full": lambda: synth.random_small(103, 2048, 12.0, 7),
    "eight_by_nodes": lambda: synth.random_small(104, 2049, 6.0, 2, weighted=False, isolated=9),
    "eight_by_cells": lambda: synth.random_small(105, 90, 8.0, 800, weighted=False),
    "eight_full": lambda: synth.random_small(106, 8192, 6.0, 9),
    "cluster_hubs": lambda: synth.random_small(107, 8800, 6.0, 11, hubs=2),
    "one_cta_weighted_k300": lambda: synth.random_small(108, 181, 9.0, 300),
    "blocks_beyond_ranks": lambda: synth.random_small(109, 1201, 9.0, 300),
    "heavy_nodes": lambda: synth.random_small(110, 3001, 6.0, 5, max_vw=(1 << 24) - 1),
    "imbalanced_input": lambda: synth.random_small(111, 3000, 5.0, 6, balanced=False),
    "long_rows_of_one_cta": _long_rows_of_one_cta,
    "largest_by_nodes": lambda: synth.random_small(112, 40000, 5.0, 2, weighted=False),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_one_launch_equals_the_oracle(upr, name):
    w = CASES[name]()
    rc0, p0, c0, _ = oracle.refine(w, w.part, rounds=4)
    for graphs in (1, 2):
        prm = upr.upr_params_default()
        prm.graphs = graphs
        ctx = upr.create_from_workload(w, params=prm)
        for call in range(3):
            p = w.part.copy()
            if rc0 != oracle.OK:
                with pytest.raises(upr.UprError):
                    upr.upr_refine(ctx, p, 4)
                continue
            st = upr.upr_refine(ctx, p, 4)
            assert np.array_equal(p, p0) and st.cut_out == c0
            if name != "imbalanced_input":                # (its repair round goes step by step)
                assert st.rebalance_graphs == st.rounds_run == 4
                # (from the second call on, graphs = 2 keeps one graph launch beyond 2^15 entries and cells)
                if graphs == 1 or call == 0 or w.m + w.n * w.k <= 1 << 15:
                    assert st.kernel_launches < 20


def test_options_and_the_edges_of_the_rule(upr):
    w = synth.random_small(120, 5000, 7.0, 6, hubs=1)
    for over, rounds in (({"append": 1}, 3), ({"lock_rebalanced": 1}, 3), ({"lp_rounds": 3}, 3),
                         ({}, 257)):
        prm = upr.upr_params_default()
        for key, val in over.items():
            setattr(prm, key, val)
        p = w.part.copy()
        st = upr.upr_refine(upr.create_from_workload(w, params=prm), p, rounds)
        rc0, p0, c0, _ = oracle.refine(w, w.part, rounds=rounds, p=oracle.params(**over))
        assert rc0 == oracle.OK and np.array_equal(p, p0) and st.cut_out == c0, (over, rounds)
    prm = upr.upr_params_default()
    prm.round_offset, prm.total_rounds = 2, 6
    p, p0 = w.part.copy(), w.part
    upr.upr_refine(upr.create_from_workload(w, params=prm), p, 3)
    for r in (3, 4, 5):
        p0 = oracle.run_round(w, p0, r, 6)[1]
    assert np.array_equal(p, p0)
    over = synth.random_small(121, 8192, 20.0, 48, weighted=False)          # just beyond 2^19
    assert over.m + over.n * over.k > 1 << 19
    p = over.part.copy()
    st = upr.upr_refine(upr.create_from_workload(over), p, 2)
    rc0, p0, c0, _ = oracle.refine(over, over.part, rounds=2)
    assert rc0 == oracle.OK and np.array_equal(p, p0) and st.cut_out == c0
