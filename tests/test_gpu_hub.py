"""Rounds whose updates go through the other side's hubs (Gram matrix of the
activeSet, quadratic form on the tensor cores, pulled rest): the oracle's tip
numbers, with the hubs covering all, most or half of the other side's edges,
hubs on the decomposed side too, and large and small activeSets."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2010_08695_gb300 as R
    R.load()
    return R


CASES = {
    # fewer middle vertices than hubs: nothing is pulled
    "all-hubs": lambda: (160_000, 200, *synth.chung_lu(160_000, 200, 250_000, 2.5, 2.4, 71)),
    # hubs of the other side and, past them, thousands of middle vertices
    "mixed": lambda: (150_001, 5_003, *synth.chung_lu(150_001, 5_003, 600_000, 2.4, 2.1, 72)),
    # vertices of very high degree on the decomposed side (the heavy ones)
    "both": lambda: (200_003, 60_000, *synth.chung_lu(200_003, 60_000, 1_200_000, 2.0, 2.1, 73)),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_hub_rounds(R, name):
    nu, nv, eu, ev = CASES[name]()
    want, _ = oracle.bup(eu, ev, nu, nv, 0)
    g = R.Graph(eu, ev, nu, nv)
    for kw in ({"P": 4}, {"P": 25}, {}):
        for mode in (False, True, -1):
            t = R.as_u64(g.tip_decompose(0, dgm=False, huc=-1, round_graphs=mode, **kw))
            assert np.array_equal(t, want), (kw, mode)
            st = g.stats()
            if mode is False:
                rounds = [(r["range"], r["frontier"], r["hi"]) for r in g.trace()]
                walked = st["peel_wedges"]
                # with full lists the per-anchor tiers alone walk exactly
                # wedges_cd wedges
                if kw != {}:
                    assert sum(walked) < st["wedges_cd"], "no round went through the hubs"
            else:
                assert rounds == [(r["range"], r["frontier"], r["hi"]) for r in g.trace()]
                assert walked == st["peel_wedges"]
        t = R.as_u64(g.tip_decompose(0, timing=True, **kw))
        assert np.array_equal(t, want), kw
        t = R.as_u64(g.tip_decompose(0, scan_frontier=-1, **kw))
        assert np.array_equal(t, want), kw


# without memory for them, the per-anchor tiers walk every round
def test_without_memory_for_hub_rounds(R):
    nu, nv, eu, ev = CASES["mixed"]()
    want, _ = oracle.bup(eu, ev, nu, nv, 0)
    g = R.Graph(eu, ev, nu, nv)
    R.receipt_optional_memory(0)
    try:
        t = R.as_u64(g.tip_decompose(0, P=4, dgm=False, huc=-1))
    finally:
        R.receipt_optional_memory(-1)
    assert np.array_equal(t, want)
    st = g.stats()
    # all wedges (those of a hybrid anchor that overflows twice)
    assert sum(st["peel_wedges"]) >= st["wedges_cd"]


def test_launches_count_the_rounds_a_tier_ran(R):
    nu, nv, eu, ev = CASES["mixed"]()
    g = R.Graph(eu, ev, nu, nv)
    g.tip_decompose(0, P=4, huc=-1, timing=True)
    st = g.stats()
    hub = sum(1 for r in g.trace() if r["ms"][1] > 0 and not any(r["ms"][t] for t in (0, 2, 3, 4)))
    assert hub > 0
    assert st["peel_launches"][1] == st["rounds_cd"]
    assert all(st["peel_launches"][t] == st["rounds_cd"] - hub for t in (0, 2, 3, 4))
