"""The fine-grained step's update lists and its two peels: the oracle's tip
numbers at the edges of what a task, a counter, a table and the list pool hold."""
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


def _check(R, eu, ev, nu, nv, Ps):
    want, _ = oracle.bup(eu, ev, nu, nv, 0)
    g = R.Graph(eu, ev, nu, nv)
    for P in Ps:
        t = R.as_u64(g.tip_decompose(0, P=P, fd_heavy_w=-1))
        assert np.array_equal(t, want), P


# supports in shared memory up to 15,360 members, list entries of 14 rank bits
# up to 16,384; a warp's 1,024 words hold 8,192 4-bit counters; short walks of
# the largest task take the table
@pytest.mark.parametrize("n", [1, 2, 31, 1024, 1025, 8192, 8193, 15360, 15361, 16384, 16385, 70000])
def test_task_edges(R, n):
    nv = max(2, n // 12)
    m = min(4 * n, n * nv // 2)
    eu, ev = synth.er(n, nv, m, seed=n) if n < 100 else \
        synth.chung_lu(n, nv, m, 2.4, 2.3, seed=n)
    _check(R, eu, ev, n, nv, (1, 3))


# groups of w members that share d keys, so counts reach the degree: 4, 8 and
# 16 bits, entries of 10 and 18 count bits; a tenth of the members has one key
# more, shared by all of them
@pytest.mark.parametrize("extra", [0, 17000])
@pytest.mark.parametrize("d,w", [(1, 513), (8, 64), (8, 65), (15, 30), (16, 30), (255, 4),
                                 (256, 4), (600, 3), (1022, 3), (1024, 3)])
def test_full_counters(R, d, w, extra):
    groups = 40
    u = np.arange(groups * w, dtype=np.int32)
    x = u[::10]
    y = np.arange(extra, dtype=np.int32)  # members with no butterfly
    eu = np.concatenate([np.repeat(u, d), x, u.size + y])
    ev = np.concatenate([np.repeat(u // w, d) * d + np.tile(np.arange(d), u.size),
                         np.full(x.size, groups * d), groups * d + 1 + y]).astype(np.int32)
    _check(R, eu.astype(np.int32), ev, u.size + extra, groups * d + 1 + extra, (1, 4))


# nearly complete: the lists of 3,200 members (10M entries) do not fit the pool
def test_lists_beyond_the_pool(R):
    n, d = 3200, 7
    u = np.arange(n, dtype=np.int32)
    deg = 2 + u % (d - 1)
    eu = np.repeat(u, deg)
    ev = np.concatenate([(k + np.arange(c)) % d for k, c in zip(u // 640, deg)]).astype(np.int32)
    _check(R, eu, ev, n, d, (1, 2))


# walks of 9,000 wedges and more in a task of 140,000 members: counters of 4 and
# 8 bits in two and four slices of a CTA's words, over ranks all along the task
def test_sliced_counters(R):
    n, hub = 140_000, 9_000
    rng = np.random.default_rng(3)
    h = rng.permutation(n)[:hub].astype(np.int64)  # members of key 0
    trio = 1 + np.arange(hub) // 3                 # a key shared by three of them
    wide = h[::10]                                 # degree 17 and more
    own = 1 + hub // 3 + np.arange(wide.size * 15)
    twin = np.arange(n) // 2 + own[-1] + 1         # pairs with one key: no butterfly
    eu = np.concatenate([h, h, np.repeat(wide, 15), np.arange(n)]).astype(np.int32)
    ev = np.concatenate([np.zeros(hub), trio, own, twin]).astype(np.int32)
    _check(R, eu, ev, n, int(ev.max()) + 1, (1,))


# supports so close together that one level sets off the next: a level then
# peels more list entries than one CTA applies in the time of a level by all
# CTAs (uniform and dense graphs, odd sizes); on power-law graphs a level peels
# a member or two
@pytest.mark.parametrize("n,nv,m,gamma,P,heavy", [
    (5_000, 20_001, 2_000_000, 0, 150, True), (6_001, 150, 300_000, 0, 150, True),
    (100_000, 30_000, 1_000_000, 2.4, 5, False),
    (20_000, 30_000, 1_000_000, 2.4, 1, False)])
def test_wide_levels_take_all_ctas(R, n, nv, m, gamma, P, heavy):
    eu, ev = synth.chung_lu(n, nv, m, gamma, gamma, 4) if gamma else synth.er(n, nv, m, 4)
    want, _ = oracle.bup(eu, ev, n, nv, 0)
    g = R.Graph(eu, ev, n, nv)
    t = R.as_u64(g.tip_decompose(0, P=P))
    assert np.array_equal(t, want)
    assert (g.stats()["fd_heavy_subsets"] > 0) == heavy


def _pool_high(reset=False):
    """Most bytes in use in the device's default memory pool since the reset."""
    import ctypes
    import torch
    cu, pool, v = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(), ctypes.c_uint64(0)
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    if reset:  # CU_MEMPOOL_ATTR_USED_MEM_HIGH
        assert cu.cuMemPoolSetAttribute(pool, 8, ctypes.byref(v)) == 0
    assert cu.cuMemPoolGetAttribute(pool, 8, ctypes.byref(v)) == 0
    return v.value


# the lists' pool follows what they can hold: a member of a dense graph has an
# entry for every other member however many wedges it walks, and power-law
# graphs an entry for six wedges or more
@pytest.mark.parametrize("nu,nv,m,gamma,P,mb", [(3_000, 3_000, 2_000_000, 0, 150, 400),
                                                (600, 2_000, 600_000, 0, 150, 150),
                                                (300_000, 90_000, 2_000_000, 2.3, 4, 600)])
def test_pool_follows_the_lists(R, nu, nv, m, gamma, P, mb):
    import torch
    eu, ev = synth.chung_lu(nu, nv, m, gamma, gamma, 6) if gamma else synth.er(nu, nv, m, 6)
    g = R.Graph(eu, ev, nu, nv)
    torch.cuda.synchronize()
    _pool_high(True)
    t = R.as_u64(g.tip_decompose(0, P=P))
    assert _pool_high() < mb << 20
    if not gamma:
        want, _ = oracle.bup(eu, ev, nu, nv, 0)
        assert np.array_equal(t, want)


@pytest.fixture
def no_optional_memory(R):
    R.receipt_optional_memory(0)
    yield
    R.receipt_optional_memory(-1)


# no memory for lists: every member walks when it is peeled, in both peels, with
# levels of one member (power law) and of thousands (uniform)
@pytest.mark.parametrize("n", [3_000, 15_360, 15_361, 40_000])
@pytest.mark.parametrize("uniform", [False, True])
def test_without_lists(R, no_optional_memory, n, uniform):
    nv = n // 12
    eu, ev = synth.er(n, nv, 4 * n, n) if uniform else synth.chung_lu(n, nv, 4 * n, 2.4, 2.3, n)
    _check(R, eu, ev, n, nv, (1, 4))


# ... and tasks whose walks outweigh their levels go to all CTAs then
def test_without_lists_long_walks_take_all_ctas(R, no_optional_memory):
    n, nv, m = 600, 2_000, 600_000
    eu, ev = synth.er(n, nv, m, 8)
    want, _ = oracle.bup(eu, ev, n, nv, 0)
    g = R.Graph(eu, ev, n, nv)
    for lists in (False, True):
        R.receipt_optional_memory(-1 if lists else 0)
        t = R.as_u64(g.tip_decompose(0))
        assert np.array_equal(t, want)
        assert (g.stats()["fd_heavy_subsets"] > 0) == (not lists)


# lists that overflow the serving engine's pool (eight entries an edge and 5M):
# a part of the members has a list, the others walk
@pytest.mark.parametrize("n,d", [(3_200, 7), (15_400, 4)])
def test_part_of_the_lists_beyond_the_pool(R, n, d):
    u = np.arange(n, dtype=np.int32)
    deg = 2 + u % (d - 1)
    eu = np.repeat(u, deg)
    ev = np.concatenate([(k + np.arange(c)) % d for k, c in zip(u // 640, deg)]).astype(np.int32)
    want, _ = oracle.bup(eu, ev, n, d, 0)
    sv = R.Server(max_inflight=1)
    rid, _ = sv.submit(eu, ev, n, d, 0)
    got = sv.wait(rid)[0]
    sv.close()
    assert np.array_equal(got, want)


# tasks whose last levels peel nearly all members go over to all CTAs there: from
# shared memory (4,000 members) and from global memory (20,000), with vertices that
# no level peels with updates, and several at once in a packed union
@pytest.mark.parametrize("n,nv,m,extra", [(4_000, 60_000, 2_400_000, 0), (4_000, 9_000, 1_200_000, 9_000),
                                          (20_000, 30_000, 3_000_000, 0)])
def test_wide_levels_are_handed_over(R, n, nv, m, extra):
    eu, ev = synth.er(n, nv, m, 12)
    y = np.arange(extra, dtype=np.int32)
    eu, ev = np.concatenate([eu, n + y]), np.concatenate([ev, nv + y // 2])
    nu, nv = n + extra, nv + extra
    want, _ = oracle.bup(eu, ev, nu, nv, 0)
    g = R.Graph(eu, ev, nu, nv)
    for P in (3, 10, 150):
        t = R.as_u64(g.tip_decompose(0, P=P))
        assert np.array_equal(t, want), P
        st, subs = g.stats(), g.subsets()
        assert st["fd_heavy_subsets"] > 0, P
        assert sum(s["levels"] for s in subs if s["heavy"]) == st["levels_fd_heavy"]
        levels = [s["levels"] for s in subs]
        t = R.as_u64(g.tip_decompose(0, P=P, fd_heavy_w=-1))
        assert np.array_equal(t, want), P
        assert g.stats()["fd_heavy_subsets"] == 0
        assert levels == [s["levels"] for s in g.subsets()], P


def test_wide_levels_of_a_union(R):
    graphs, wants = [], []
    for i in range(3):
        n, nv, m = 3_500 + 500 * i, 12_000, 900_000
        eu, ev = synth.er(n, nv, m, 40 + i)
        graphs.append(R.Graph(eu, ev, n, nv))
        wants.append(oracle.bup(eu, ev, n, nv, 0)[0])
    outs = R.receipt_decompose_batch(graphs, [0] * 3, P=4)
    for o, w in zip(outs, wants):
        assert np.array_equal(R.as_u64(o), w)


# many equal dense tasks: their estimated costs are equal too
def test_equal_dense_tasks(R):
    eu, ev = synth.er(400, 300, 30_000, 3)
    want, _ = oracle.bup(eu, ev, 400, 300, 0)
    g = R.Graph(eu, ev, 400, 300)
    for k in (2, 17, 64, 150):
        for P in (1, 5, 150):
            for t in R.receipt_decompose_batch([g] * k, [0] * k, P=P):
                assert np.array_equal(R.as_u64(t), want), (k, P)
