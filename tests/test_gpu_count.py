"""Butterfly counts at the edges of the counting tiers: start points of degree
around the bit-sliced part's classes (one warp, one CTA, several CTAs), end
points on both sides of its 1,024 keys, tails of every size past them, and the
start points of a packed union (whose keys begin at their own graph)."""
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


def _with_degrees(nu, nv, degs, m, seed):
    """`degs[i]` random neighbours of V vertex i, `m` uniform edges elsewhere."""
    rng = np.random.default_rng(seed)
    eu = [rng.choice(nu, d, replace=False) for d in degs]
    ev = [np.full(d, i) for i, d in enumerate(degs)]
    ru, rv = synth.er(nu, nv - len(degs), m, seed)
    return np.concatenate(eu + [ru]).astype(np.int32), \
        np.concatenate(ev + [rv + len(degs)]).astype(np.int32)


def _check(R, eu, ev, nu, nv, noalloc):
    import torch
    cu, cv = oracle.count_vp(eu, ev, nu, nv)
    g = R.Graph(eu, ev, nu, nv)
    gu, gv = g.count_butterflies()
    assert np.array_equal(R.as_u64(gu), cu) and np.array_equal(R.as_u64(gv), cv)
    if noalloc:
        gu.fill_(-1), gv.fill_(-1)
        R.receipt_count_butterflies_noalloc(g.handle, gu, gv)
        torch.cuda.synchronize()
        assert np.array_equal(R.as_u64(gu), cu) and np.array_equal(R.as_u64(gv), cv)


@pytest.mark.parametrize("degs", [
    (1, 2, 3, 7, 8, 9, 31, 32, 33),
    (255, 256, 257, 511, 512, 513, 1023, 1024, 1025),
    (8191, 8192, 8193, 16384, 16385, 24999, 25000),
])
def test_degree_classes(R, degs):
    nu, nv = 25_000, 2_000
    eu, ev = _with_degrees(nu, nv, degs * 3, 150_000, 5)
    _check(R, eu, ev, nu, nv, True)
    _check(R, ev, eu, nv, nu, True)


@pytest.mark.parametrize("nu,nv,m", [(1024, 1025, 60_000), (1500, 1023, 200_000), (6000, 5500, 900_000),
                                     (60_000, 3_000, 900_000), (300_000, 90_000, 900_000)])
def test_tails(R, nu, nv, m):
    # uniform edges: most end points lie past the first 1,024
    eu, ev = synth.er(nu, nv, m, 9)
    _check(R, eu, ev, nu, nv, max(nu, nv) <= 65536)


def test_union_counts_from_its_own_first_key(R):
    graphs, wants = [], []
    for i in range(6):
        nu, nv, m = 3000 + 700 * i, 1500 + 100 * i, 30_000
        eu, ev = synth.chung_lu(nu, nv, m, 2.2, 2.2, 30 + i)
        graphs.append(R.Graph(eu, ev, nu, nv))
        wants.append(oracle.bup(eu, ev, nu, nv, i % 2)[0])
    outs = R.receipt_decompose_batch(graphs, [i % 2 for i in range(6)])
    st = graphs[0].stats()
    for o, w in zip(outs, wants):
        assert np.array_equal(R.as_u64(o), w)
    # no start point needs the global counters
    assert st["count_points"][3] == 0 and st["count_points"][4] == 0


# hubs whose end points nearly all come after them: degrees on both sides of the
# steps that each tier takes (32, 64, 256, 512 middle points a step, 8 steps), with
# a few wedges (other hubs' common neighbours) and with many
@pytest.mark.parametrize("nu,m", [(70_000, 30_000), (120_000, 400_000)])
def test_hubs_of_few_wedges(R, nu, m):
    degs = [d + k for d in (255, 512, 2048, 4096, 9000, 20_000, 30_000) for k in (0, 1)]
    eu, ev = _with_degrees(nu, 20_000, degs, m, 7)
    _check(R, eu, ev, nu, 20_000, False)
    # ... and of degree 65,535 and more
    eu, ev = _with_degrees(nu, 20_000, [300, 65_534, 65_535, 65_536, 66_000], m, 8)
    _check(R, eu, ev, nu, 20_000, False)


def test_hubs_of_few_wedges_without_allocations(R):
    degs = [d + k for d in (255, 512, 2048, 4096, 9000, 30_000, 65_533) for k in (0, 1)]
    eu, ev = _with_degrees(65_536, 9_000, degs, 60_000, 9)
    _check(R, eu, ev, 65_536, 9_000, True)
