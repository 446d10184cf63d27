"""Calls at the limits of the team launches, against the oracle: block counts
where a kernel's shared memory ends."""
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


def _params(upr, **over):
    p = upr.upr_params_default()
    for key, val in over.items():
        setattr(p, key, val)
    return p


def _refined_as_the_oracle(upr, ctx, w, rounds=3, calls=1):
    rc, p0, c0, _ = oracle.refine(w, w.part, rounds=rounds)
    assert rc == oracle.OK
    for _ in range(calls):
        p = w.part.copy()
        st = upr.upr_refine(ctx, p, rounds)
        assert np.array_equal(p, p0) and st.cut_out == c0
    return st


@pytest.mark.parametrize("graphs", [1, 2])
@pytest.mark.parametrize("n,k,weighted", [(1000, k, True) for k in (318, 319, 320, 322, 323)] +
                         [(700, k, False) for k in (639, 640, 645, 646)])
def test_small_graph_where_the_buckets_stop_fitting(upr, n, k, weighted, graphs):
    """The buckets of a small graph's one launch: 584 k bytes of shared memory
    with node weights, 292 k without, beside the kernel's static part."""
    w = synth.random_small(7, n, 8.0, k, weighted=weighted)
    assert w.m + n * k <= 1 << 19
    ctx = upr.create_from_workload(w, params=_params(upr, graphs=graphs))
    _refined_as_the_oracle(upr, ctx, w, calls=2)


AFTER_A_FAILED_CALL = r"""
import sys
sys.path.insert(0, {root!r})
import numpy as np, torch
import oracle, synth
import paper_2308_15494_gb300 as upr

def valid(k):
    w = synth.random_small(9, 900, 6.0, k)
    ctx = upr.create_from_workload(w)
    p = w.part.copy()
    st = upr.upr_refine(ctx, p, 3)
    rc, p0, c0, _ = oracle.refine(w, w.part, rounds=3)
    assert rc == oracle.OK and np.array_equal(p, p0) and st.cut_out == c0
    return ctx, w

kept, w = valid(5)                         # (everything is loaded and warm)
graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
x = torch.zeros(8, device="cuda")
status = None
try:
    with torch.cuda.stream(side):
        graph.capture_begin(capture_error_mode="global")
        x.add_(1)
        try:                               # allocates: refused while the thread captures
            upr.create_from_workload(w)
        except upr.UprError as e:
            status = e.status
        graph.capture_end()
except RuntimeError:                       # (the refused call has ended the capture)
    pass
assert status in (upr.UPR_ERR_CUDA, upr.UPR_ERR_OOM), status
p = w.part.copy()
upr.upr_refine(kept, p, 3)                 # a kept context, then a new one
valid(7)
print("ok")
"""


def test_a_failed_call_leaves_the_next_one_alone(upr):
    """A call that a CUDA error ends (here: an allocation that the runtime
    refuses during a stream capture) does not fail the calls after it."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", AFTER_A_FAILED_CALL.format(root=root)], cwd=root, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-2000:]


@pytest.mark.parametrize("graphs", [0, 1, 2])
def test_a_barrier_that_gives_up_stops_every_step(upr, graphs):
    """A grid barrier that one CTA never reaches: the wait runs out and no CTA
    goes past it.  The context's next calls then end with an error status, the
    partition as it was, in every form of the rounds (launched one by one, the
    rebalancing loops or the whole call as captured graphs), and a binding
    brings the context back."""
    w = synth.random_small(73, 70000, 5.0, 6, hubs=1)
    ctx = upr.create_from_workload(w, params=_params(upr, graphs=graphs))
    _refined_as_the_oracle(upr, ctx, w, calls=4)
    ctas, passed = upr.upr_debug_barrier(ctx, 0)
    assert ctas > 16 and passed == ctas
    ctas, passed = upr.upr_debug_barrier(ctx, 1)
    assert passed == 0
    for _ in range(2):
        p = w.part.copy()
        with pytest.raises(upr.UprError) as e:
            upr.upr_refine(ctx, p, 3)
        assert e.value.status == upr.UPR_ERR_CUDA and np.array_equal(p, w.part)
    upr.upr_rebind(ctx, w.xadj, w.adj, w.k, w.eps, vwgt=w.vwgt, adjw=w.adjw)
    _refined_as_the_oracle(upr, ctx, w, calls=3)


def test_a_batch_whose_barrier_gave_up(upr):
    ws = [synth.random_small(74 + i, 18000, 5.0, 6) for i in range(4)]
    ctx = upr.create_batch_from_workloads(ws)
    part0 = np.concatenate([w.part for w in ws]).astype(np.int32)
    p = part0.copy()
    status, _, cut, _ = upr.upr_batch_refine(ctx, p, 3)
    assert upr.upr_debug_barrier(ctx, 2)[1] == 0
    q = part0.copy()
    with pytest.raises(upr.UprError) as e:
        upr.upr_batch_refine(ctx, q, 3)
    assert e.value.status == upr.UPR_ERR_CUDA and np.array_equal(q, part0)
    upr.upr_batch_rebind(ctx, [(w.xadj, w.adj, w.vwgt, w.adjw) for w in ws], [w.k for w in ws], [w.eps for w in ws])
    q = part0.copy()
    upr.upr_batch_refine(ctx, q, 3)
    assert np.array_equal(q, p)
    for i, w in enumerate(ws):
        rc, p0, c0, _ = oracle.refine(w, w.part, rounds=3)
        a, b = ctx.offsets[i], ctx.offsets[i + 1]
        assert rc == status[i] == 0 and np.array_equal(p[a:b], p0) and cut[i] == c0


def test_a_small_team_has_no_grid_barrier(upr):
    ctx = upr.create_from_workload(synth.random_small(75, 5000, 5.0, 6))
    with pytest.raises(upr.UprError) as e:
        upr.upr_debug_barrier(ctx, 0)
    assert e.value.status == upr.UPR_ERR_INVALID


@pytest.mark.parametrize("k,deg", [(8, 3.0), (128, 9.0), (256, 9.0)])
def test_dense_rounds_after_hashed_rows_ran_out(upr, k, deg):
    """Rows of min(k, deg) + 1 slots run out and the binding goes on with the
    dense table, on tiles of its own (512 rows at k = 8, 32 at k = 256): results,
    a later call's and the table itself as the oracle's; a binding after it
    starts on hashed rows again."""
    w = synth.random_small(76 + k, 9000, deg, k, hubs=1)
    ctx = upr.create_from_workload(w, params=_params(upr, table=3))
    for _ in range(2):
        st = _refined_as_the_oracle(upr, ctx, w, calls=2)
        assert st.sparse_table == 0
        W, _ = upr.upr_debug_gain_table(ctx, w.part)
        assert np.array_equal(W, oracle.gain_table(w, w.part)[0])
        upr.upr_rebind(ctx, w.xadj, w.adj, w.k, w.eps, vwgt=w.vwgt, adjw=w.adjw)
        W, _ = upr.upr_debug_gain_table(ctx, w.part)          # (from the hashed rows)
        assert np.array_equal(W, oracle.gain_table(w, w.part)[0])


def test_label_propagation_falls_back_from_hashed_rows(upr):
    w = synth.random_small(77, 9000, 9.0, 128)
    ctx = upr.create_from_workload(w, params=_params(upr, table=3, lp_rounds=4))
    rc, p0, c0, _ = oracle.refine(w, w.part, rounds=3, p=oracle.params(lp_rounds=4))
    for _ in range(2):
        p = w.part.copy()
        st = upr.upr_refine(ctx, p, 3)
        assert np.array_equal(p, p0) and st.cut_out == c0
    assert st.sparse_table == 0


@pytest.mark.parametrize("bits", [30, 31, 32])
@pytest.mark.parametrize("k", [4, 24, 64])
def test_packed_scores_at_their_width(upr, k, bits):
    """Unit node weights and edge weights so heavy that the largest omega(I(v))
    and a column index take `bits` bits together: the selection packs a score
    and its column into one integer up to 30, the proposals up to 31."""
    w = synth.random_small(78 + k, 3000, 8.0, k, weighted=False, hubs=1, balanced=False)
    gb = bits - max(1, (k - 1).bit_length())
    adjw = synth.edge_weights_uniform(w.xadj, w.adj, 1, 16, 5).astype(np.int64)
    heaviest = max(int(adjw[w.xadj[v]:w.xadj[v + 1]].sum()) for v in range(w.n))
    adjw *= ((1 << gb) - 1) // heaviest
    heaviest = max(int(adjw[w.xadj[v]:w.xadj[v + 1]].sum()) for v in range(w.n))
    assert heaviest.bit_length() == gb
    w.adjw = adjw.astype(np.int32)
    ctx = upr.create_from_workload(w, params=_params(upr, graphs=0))       # (the rounds launched step by step)
    st = _refined_as_the_oracle(upr, ctx, w)
    assert st.repaired_input == 1 and st.n_rebalance_moves > 0 and st.n_moves > 0
    rc, p, t = upr.upr_debug_round(ctx, w.part, 0, 2, rebalance_only=True)
    rc0, p0, _, o = oracle.run_round(w, w.part, 0, 2, rebalance_only=True)
    assert rc == rc0 == 0 and np.array_equal(p, p0)
    _compare_traces(t, o)
    rc, p, t = upr.upr_debug_round(ctx, p0, 1, 2)
    rc0, p1, _, o = oracle.run_round(w, p0, 1, 2)
    assert rc == rc0 == 0 and np.array_equal(p, p1)
    _compare_traces(t, o)
