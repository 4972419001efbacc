"""The build at the edges of its sorts and tiles: one vertex a side, label bits
around a digit's ten, tiles of 1,024, 2,048 and 4,096 keys, duplicates across
them, and hubs on the side whose degrees are counted."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2010_08695_gb300 as R
    R.load()
    return R


@pytest.mark.parametrize("nu,nv,m", [
    (1, 1, 1), (1, 5000, 4000), (5000, 1, 4000), (2, 1025, 1024), (1024, 1024, 2048),
    (1025, 1023, 2049), (33, 70000, 16385), (70000, 33, 16384), (1 << 20, 3, 1000),
    (300_000, 900_000, (1 << 21) - 1), (300_000, 900_000, (1 << 21) + 4097)])
@pytest.mark.parametrize("dup", [False, True])
def test_sizes(R, nu, nv, m, dup):
    rng = np.random.default_rng(m)
    if dup:
        eu, ev = rng.integers(0, nu, m), rng.integers(0, nv, m)
        ev[: m // 4] = 0  # a hub, and runs of equal edges
        eu[: m // 8] %= 3
    else:
        k = np.unique(rng.integers(0, nu * nv, m))
        rng.shuffle(k)
        eu, ev = k // nv, k % nv
    eu, ev = eu.astype(np.int32), ev.astype(np.int32)
    key = np.unique(eu.astype(np.int64) * nv + ev)
    g = R.Graph(eu, ev, nu, nv)
    assert g.m == key.size
    if not dup:
        R.Graph(eu, ev, nu, nv, dedup=False)
    cu, cv = oracle.count_vp((key // nv).astype(np.int32), (key % nv).astype(np.int32), nu, nv)
    gu, gv = g.count_butterflies()
    assert np.array_equal(R.as_u64(gu), cu) and np.array_equal(R.as_u64(gv), cv)
