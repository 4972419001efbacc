"""The coarse-grained step in one cooperative launch (sides whose keys fit a few
dense windows): the same tip numbers as the oracle and the same rounds as the
per-round kernels, at the edges of its windows and of its records."""
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


def _rounds(g):
    return [(r["range"], r["frontier"], r["hi"]) for r in g.trace()]


# one dense window has 36,864 keys, at most four windows; the last side takes
# the per-round kernels
@pytest.mark.parametrize("n", [1, 33, 2049, 36864, 36865, 73729, 147456, 147457])
def test_window_edges(R, n):
    nv = max(2, n // 40)
    m = min(3 * n, n * nv // 2)
    eu, ev = synth.er(n, nv, m, seed=n) if n < 100 else \
        synth.chung_lu(n, nv, m, 2.4, 2.3, seed=n)
    want, _ = oracle.bup(eu, ev, n, nv, 0)
    g = R.Graph(eu, ev, n, nv)
    for kw in ({}, {"P": 3}, {"dgm": False}, {"dgm_frac_1024": 8}, {"warp_max_w": 16}):
        t = R.as_u64(g.tip_decompose(0, **kw))
        assert np.array_equal(t, want), kw
        recs = _rounds(g)
        t = R.as_u64(g.tip_decompose(0, round_graphs=-1, **kw))
        assert np.array_equal(t, want), kw
        assert recs == _rounds(g), kw


def test_more_rounds_than_one_launch_records(R):
    # a ladder: u_i shares one butterfly with each neighbour, so below the
    # bound 2 the peel cascades in from both ends, two vertices a round
    k = 9000
    i = np.arange(k, dtype=np.int32)
    eu = np.repeat(i, 4)
    ev = np.stack([i, i + 1, k + 1 + i, k + 2 + i], axis=1).reshape(-1).astype(np.int32)
    want, _ = oracle.bup(eu, ev, k, 2 * (k + 1), 0)
    g = R.Graph(eu, ev, k, 2 * (k + 1))
    t = R.as_u64(g.tip_decompose(0, P=20000))
    assert np.array_equal(t, want)
    assert g.stats()["rounds_cd"] > 4096
    recs = _rounds(g)
    t = R.as_u64(g.tip_decompose(0, P=20000, round_graphs=-1))
    assert np.array_equal(t, want) and recs == _rounds(g)


# short walks counted by groups of warps: degrees around the 4-, 8- and 16-bit
# counters, members with d keys shared by w of them, in one and several windows
@pytest.mark.parametrize("pad", [0, 40_000, 200_000])
@pytest.mark.parametrize("d,w", [(2, 300), (15, 40), (16, 40), (255, 5), (256, 5), (1024, 2)])
def test_short_walks(R, d, w, pad):
    groups = 30
    u = np.arange(groups * w)
    x = u[::7]  # one more key, shared by them all
    y = np.arange(pad)  # pairs without a butterfly
    rng = np.random.default_rng(d)
    lab = rng.permutation(u.size + pad)
    eu = lab[np.concatenate([np.repeat(u, d), x, u.size + y])].astype(np.int32)
    ev = np.concatenate([np.repeat(u // w, d) * d + np.tile(np.arange(d), u.size),
                         np.full(x.size, groups * d), groups * d + 1 + y // 2]).astype(np.int32)
    nv = int(ev.max()) + 1
    want, _ = oracle.bup(eu, ev, u.size + pad, nv, 0)
    g = R.Graph(eu, ev, u.size + pad, nv)
    for kw in ({}, {"P": 4}, {"dgm_frac_1024": 8}, {"warp_max_w": 16}):
        t = R.as_u64(g.tip_decompose(0, **kw))
        assert np.array_equal(t, want), kw
        recs = _rounds(g)
        t = R.as_u64(g.tip_decompose(0, round_graphs=-1, **kw))
        assert np.array_equal(t, want), kw
        assert recs == _rounds(g), kw


# updates by lists made beforehand, counters of 16 bits in slices of a CTA's
# words; two windows' keys are the most a listed side has
@pytest.mark.parametrize("n", [3000, 40_000, 73_728, 73_729])
def test_lists_of_hubs(R, n):
    nv, hubs, deg = 2000, 40, 600
    rng = np.random.default_rng(n)
    hu = rng.choice(n, hubs, replace=False)
    ru, rv = synth.er(n, nv, 2 * n, seed=n)
    eu = np.concatenate([np.repeat(hu, deg), ru]).astype(np.int32)
    ev = np.concatenate([rng.choice(nv, deg, replace=False) for _ in range(hubs)] + [rv]).astype(np.int32)
    key = np.unique(eu.astype(np.int64) * nv + ev)
    eu, ev = (key // nv).astype(np.int32), (key % nv).astype(np.int32)
    want, _ = oracle.bup(eu, ev, n, nv, 0)
    g = R.Graph(eu, ev, n, nv)
    for kw in ({}, {"P": 5}, {"huc": -1}):
        t = R.as_u64(g.tip_decompose(0, **kw))
        assert np.array_equal(t, want), kw
        recs = _rounds(g)
        t = R.as_u64(g.tip_decompose(0, round_graphs=-1, **kw))
        assert np.array_equal(t, want), kw
        assert recs == _rounds(g), kw


# without memory for lists, the other two forms of one window: windows, and
# groups of warps (short walks); the same counters as the per-round kernels
@pytest.mark.parametrize("lists", [True, False])
@pytest.mark.parametrize("n,nv,per,gamma", [(1, 2, 1, 0), (33, 2, 1, 0), (2_049, 51, 3, 2.4),
                                            (36_864, 921, 3, 2.4), (36_864, 20_000, 4, 0),
                                            (20_000, 5_000, 10, 2.3)])
def test_one_window_forms(R, n, nv, per, gamma, lists):
    m = min(per * n, n * nv // 2)
    eu, ev = synth.chung_lu(n, nv, m, gamma, gamma, n) if gamma else synth.er(n, nv, m, n)
    want, _ = oracle.bup(eu, ev, n, nv, 0)
    g = R.Graph(eu, ev, n, nv)
    for kw in ({}, {"P": 3}, {"dgm": False}, {"dgm_frac_1024": 8}, {"warp_max_w": 16}):
        R.receipt_optional_memory(-1 if lists else 0)
        try:
            t = R.as_u64(g.tip_decompose(0, **kw))
        finally:
            R.receipt_optional_memory(-1)
        assert np.array_equal(t, want), kw
        recs, st = _rounds(g), g.stats()
        t = R.as_u64(g.tip_decompose(0, round_graphs=-1, **kw))
        assert np.array_equal(t, want), kw
        assert recs == _rounds(g), kw
        per_round = g.stats()
        if per_round["peel_anchors"][1]:
            continue  # hub rounds, which walk less
        for k in ("peel_wedges", "peel_mids", "peel_anchors", "peel_pairs"):
            assert sum(st[k]) == sum(per_round[k]), (kw, k)


# a packed union by windows
def test_union_by_windows(R):
    graphs, wants = [], []
    for i in range(5):
        nu, nv, m = 36_864 - 9_000 * i, 2_000 + 300 * i, 90_000
        eu, ev = synth.chung_lu(nu, nv, m, 2.3, 2.3, 60 + i)
        graphs.append(R.Graph(eu, ev, nu, nv))
        wants.append(oracle.bup(eu, ev, nu, nv, i % 2)[0])
    R.receipt_optional_memory(0)
    try:
        outs = R.receipt_decompose_batch(graphs, [i % 2 for i in range(5)])
    finally:
        R.receipt_optional_memory(-1)
    for o, w in zip(outs, wants):
        assert np.array_equal(R.as_u64(o), w)


# anchors whose walks may be long are fetched fewer at a time (8, 6, 1): the
# CTAs that have none left wait for the last fetch
@pytest.mark.parametrize("ds,do", [(1_000, 10_000), (40_000, 10_000), (60_000, 25_000)])
def test_anchors_per_fetch(R, ds, do):
    n, nv = 26_001, 61_000
    rng = np.random.default_rng(do)
    ru, rv = synth.er(n, nv, 4 * n, do)
    eu = np.concatenate([np.full(ds, 7), rng.choice(n, do, replace=False), ru]).astype(np.int64)
    ev = np.concatenate([rng.choice(nv, ds, replace=False), np.full(do, 5), rv]).astype(np.int64)
    key = np.unique(eu * nv + ev)
    eu, ev = (key // nv).astype(np.int32), (key % nv).astype(np.int32)
    want, _ = oracle.bup(eu, ev, n, nv, 0)
    g = R.Graph(eu, ev, n, nv)
    for kw in ({}, {"P": 3}, {"huc": -1}):
        R.receipt_optional_memory(0)
        try:
            t = R.as_u64(g.tip_decompose(0, **kw))
        finally:
            R.receipt_optional_memory(-1)
        assert np.array_equal(t, want), kw
        recs = _rounds(g)
        t = R.as_u64(g.tip_decompose(0, round_graphs=-1, **kw))
        assert np.array_equal(t, want), kw
        assert recs == _rounds(g), kw


# a vertex whose counts do not fit above the 17 rank bits of a side of more than
# 65,536: no lists (degree 32,768 and more), and the edge below it
@pytest.mark.parametrize("n", [65_536, 65_537, 73_728])
@pytest.mark.parametrize("deg", [32_767, 32_768])
def test_degrees_past_a_list_entry(R, n, deg):
    nv = 33_000
    rng = np.random.default_rng(n + deg)
    ru, rv = synth.er(n, nv, 3 * n, n)
    keep = ru != 9
    eu = np.concatenate([np.full(deg, 9), ru[keep]]).astype(np.int32)
    ev = np.concatenate([rng.choice(nv, deg, replace=False), rv[keep]]).astype(np.int32)
    want, _ = oracle.bup(eu, ev, n, nv, 0)
    g = R.Graph(eu, ev, n, nv)
    assert g.max_degree[0] == deg
    for kw in ({}, {"P": 4}):
        t = R.as_u64(g.tip_decompose(0, **kw))
        assert np.array_equal(t, want), kw
        recs = _rounds(g)
        t = R.as_u64(g.tip_decompose(0, round_graphs=-1, **kw))
        assert np.array_equal(t, want), kw
        assert recs == _rounds(g), kw
