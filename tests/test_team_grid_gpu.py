"""The team launches at the edges of their sizes, against the oracle: one CTA up
to 2048 nodes, a cluster of at most 16 up to 65536, beyond a cooperative grid
with a grid barrier.  On the grid: every form of the ordered phases (blocks
ranked by warp sums up to 256 of them, sorted beyond; selection items of 32 and
64 bits; rebalancing keys of one word and of 128 bits; appended sequences, the
oscillation guard, batches), which smaller cases reach on clusters only."""
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


def _skewed(seed, k, weighted=True, max_vw=8, max_ew=9):
    """An R-MAT graph of 2^17 nodes (128 CTAs), whose rounds overload blocks."""
    xadj, adj = synth.rmat(17, 5, 0.57, 0.19, 0.19, seed)
    n = len(xadj) - 1
    rng = np.random.Generator(np.random.PCG64(seed))
    if not weighted:
        return synth.Workload(f"skewed{seed}", n, xadj, adj, None, None, k, 0.03,
                              synth.part_random_balanced(n, k, seed), 3)
    vwgt = rng.integers(1, max_vw + 1, size=n, dtype=np.int32)
    order = rng.permutation(n)
    order = order[np.argsort(-vwgt[order], kind="stable")]          # dealt heaviest first, back and forth
    pos = np.arange(n) % (2 * k)
    part = np.empty(n, np.int32)
    part[order] = np.where(pos < k, pos, 2 * k - 1 - pos)
    return synth.Workload(f"skewed{seed}", n, xadj, adj, synth.edge_weights_uniform(xadj, adj, 1, max_ew, seed),
                          vwgt, k, 0.03, part, 3)


CASES = {
    "one_cta_last": lambda: synth.random_small(301, 2048, 6.0, 5, hubs=1),
    "cluster_first": lambda: synth.random_small(302, 2049, 6.0, 5, hubs=1),
    "cluster_last": lambda: synth.random_small(303, 65536, 4.0, 6, weighted=False),
    "grid_first": lambda: synth.random_small(304, 65537, 4.0, 6, weighted=False),
    "grid_ranked_blocks": lambda: _skewed(305, 256),
    "grid_sorted_blocks": lambda: _skewed(306, 257),
    "grid_sorted_blocks_unit": lambda: _skewed(307, 300, weighted=False),
    "grid_wide_items": lambda: _skewed(308, 11, max_ew=1 << 18),
    "grid_wide_keys": lambda: _skewed(309, 8, max_vw=(1 << 21) - 1, max_ew=1 << 17),
    "grid_wide_keys_sorted": lambda: _skewed(310, 270, max_vw=(1 << 21) - 1, max_ew=1 << 17),
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
    if w.n > 65536:
        ctas, passed = upr.upr_debug_barrier(ctx, 0)      # (a grid barrier, whole)
        assert passed == ctas == min(-(-w.n // 1024), ctas)


@pytest.mark.parametrize("over", [{"append": 1}, {"lock_rebalanced": 1}, {"gain_priority": 1}, {"graphs": 0}])
def test_options_on_the_grid(upr, over):
    w = _skewed(311, 9)
    prm = upr.upr_params_default()
    for key, val in over.items():
        setattr(prm, key, val)
    of_oracle = {key: val for key, val in over.items() if key != "graphs"}
    rc0, p0, c0, _ = oracle.refine(w, w.part, rounds=3, p=oracle.params(**of_oracle))
    ctx = upr.create_from_workload(w, params=prm)
    for _ in range(2):
        p = w.part.copy()
        st = upr.upr_refine(ctx, p, 3)
        assert rc0 == oracle.OK and np.array_equal(p, p0) and st.cut_out == c0


@pytest.mark.parametrize("count,n,k", [(4, 18000, 5), (300, 240, 64)])
def test_batch_on_the_grid(upr, count, n, k):
    """A few graphs, and so many that their blocks have no prefilter (more than
    2^14 of them); every fifth input is imbalanced."""
    ws = [synth.random_small(320 + i, n + 3 * i, 5.0, k, balanced=i % 5 != 4) for i in range(count)]
    ctx = upr.create_batch_from_workloads(ws)
    assert ctx.n > 65536
    part = np.concatenate([w.part for w in ws]).astype(np.int32)
    status, _, cut, _ = upr.upr_batch_refine(ctx, part, 3)
    for i, w in enumerate(ws):
        rc0, p0, c0, _ = oracle.refine(w, w.part, rounds=3)
        a, b = ctx.offsets[i], ctx.offsets[i + 1]
        if rc0 == oracle.OK:
            assert status[i] == 0 and np.array_equal(part[a:b], p0) and cut[i] == c0, i
        else:
            assert status[i] == upr.UPR_ERR_INFEASIBLE and np.array_equal(part[a:b], w.part), i


@pytest.mark.parametrize("n,k,weighted", [(1500, 4, True), (3000, 7, False), (9000, 12, True)])
def test_small_graphs_by_one_launch_and_step_by_step(upr, n, k, weighted):
    """The two forms of a small graph's rounds: few launches with graphs = 1 (one
    of them the rounds), many with graphs = 0; the same results."""
    w = synth.random_small(330 + k, n, 6.0, k, weighted=weighted, hubs=1)
    rc0, p0, c0, _ = oracle.refine(w, w.part, rounds=3)
    launches = []
    for graphs in (1, 0):
        prm = upr.upr_params_default()
        prm.graphs = graphs
        p = w.part.copy()
        st = upr.upr_refine(upr.create_from_workload(w, params=prm), p, 3)
        assert rc0 == oracle.OK and np.array_equal(p, p0) and st.cut_out == c0
        launches.append(st.kernel_launches)
    assert launches[0] <= 4 < 30 < launches[1]


@pytest.mark.parametrize("shift", [1, 2, 3])
def test_cut_of_an_adjacency_at_any_alignment(upr, shift):
    """Adjacency and weights that start 4, 8 or 12 bytes behind a 16-byte
    boundary are read entry by entry."""
    import torch
    w = synth.random_small(340, 5000, 9.0, 6, hubs=1)

    def dev(a, off):
        if a is None:
            return None
        t = torch.zeros(len(a) + off, dtype=torch.from_numpy(a[:1].copy()).dtype, device="cuda")
        t[off:] = torch.from_numpy(np.ascontiguousarray(a))
        return t[off:]

    adj = dev(w.adj, shift)
    assert adj.data_ptr() % 16 == 4 * shift
    c, bw = upr.upr_cut_noalloc(dev(w.xadj, 0), adj, dev(w.part, 0), w.k, vwgt=dev(w.vwgt, shift),
                                adjw=dev(w.adjw, 4 - shift))
    c0, bw0 = oracle.cut(w, w.part)
    assert c == c0 and np.array_equal(bw, bw0)
    bad = w.adj.copy()
    bad[-1] = w.n
    with pytest.raises(upr.UprError) as e:
        upr.upr_cut_noalloc(dev(w.xadj, 0), dev(bad, shift), dev(w.part, 0), w.k)
    assert e.value.status == upr.UPR_ERR_INVALID
