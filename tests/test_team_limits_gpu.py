"""Calls at the limits of the team launches, against the oracle: block counts
where a kernel's shared memory ends."""
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
