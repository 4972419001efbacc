"""Calls in little device memory: work space that only saves time is left out."""
import contextlib
import ctypes

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


@contextlib.contextmanager
def memory_left(mb):
    """All but `mb` MB of the device's free memory is taken (what the library's
    pool holds unused counts as free)."""
    import torch
    cu, pool = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p()
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    assert cu.cuMemPoolTrimTo(pool, ctypes.c_size_t(0)) == 0
    taken = [torch.empty(torch.cuda.mem_get_info()[0] - (mb << 20), dtype=torch.uint8,
                         device="cuda")]
    try:
        yield
    finally:
        taken.clear()
        torch.cuda.empty_cache()


# 2M + 2M vertices: 512 MB of masks, the rest of a count about 260 MB
def test_count_without_masks(R):
    import torch
    nu = nv = 2_000_000
    eu, ev = synth.chung_lu(nu, nv, 4_000_000, 2.4, 2.4, 3)
    g = R.Graph(eu, ev, nu, nv)
    cu, cv = g.count_butterflies()
    du, dv = torch.empty_like(cu), torch.empty_like(cv)
    with memory_left(420):
        R.receipt_count_butterflies(g.handle, du, dv)
        torch.cuda.synchronize()
    assert torch.equal(cu, du) and torch.equal(cv, dv)


@pytest.mark.parametrize("nu,nv,m,gamma", [(1, 1, 1, 0), (1025, 1023, 50_000, 0), (3_000, 700, 60_000, 2.2),
                                           (40_000, 9_000, 300_000, 2.1), (20_000, 200, 400_000, 0)])
def test_counts_without_optional_memory(R, nu, nv, m, gamma):
    eu, ev = synth.chung_lu(nu, nv, m, gamma, gamma, 5) if gamma else synth.er(nu, nv, m, 5)
    cu, cv = oracle.count_vp(eu, ev, nu, nv)
    g = R.Graph(eu, ev, nu, nv)
    R.receipt_optional_memory(0)
    try:
        gu, gv = g.count_butterflies()
        t = R.receipt_decompose_batch([g, g, g], [0, 1, 0])
    finally:
        R.receipt_optional_memory(-1)
    assert np.array_equal(R.as_u64(gu), cu) and np.array_equal(R.as_u64(gv), cv)
    want = [oracle.bup(eu, ev, nu, nv, i)[0] for i in (0, 1)]
    for i, w in enumerate((want[0], want[1], want[0])):
        assert np.array_equal(R.as_u64(t[i]), w)


# memory that the library's pool keeps unused is there for a recount
def test_recount_in_memory_kept_by_the_pool(R):
    import torch
    nu, nv = 200_000, 60_000
    eu, ev = synth.chung_lu(nu, nv, 600_000, 2.4, 2.2, 4)
    g = R.Graph(eu, ev, nu, nv)
    want = R.as_u64(g.tip_decompose(0))
    cu, p = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p()
    with memory_left(1300):
        assert cu.cuMemAllocAsync(ctypes.byref(p), ctypes.c_size_t(1100 << 20), ctypes.c_void_p(0)) == 0
        assert cu.cuMemFreeAsync(p, ctypes.c_void_p(0)) == 0
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] < 300 << 20
        out = torch.empty(nu, dtype=torch.int64, device="cpu").to("cuda")
        t = R.as_u64(g.tip_decompose(0, huc_factor_1024=1, out=out))
    assert np.array_equal(t, want)
    assert g.stats()["huc_recounts"] > 0


# ... and a recount that does not fit is left out (the global tier's counters
# alone: 8 bytes a vertex and SM)
def test_recount_without_memory(R):
    nu, nv = 1_000_000, 60_000
    eu, ev = synth.chung_lu(nu, nv, 1_000_000, 2.4, 2.2, 4)
    g = R.Graph(eu, ev, nu, nv)
    want = R.as_u64(g.tip_decompose(0, huc_factor_1024=1))
    assert g.stats()["huc_recounts"] > 0
    with memory_left(900):
        t = R.as_u64(g.tip_decompose(0, huc_factor_1024=1))
    assert np.array_equal(t, want)
    assert g.stats()["huc_recounts"] == 0


# counting's masks (132 bytes a vertex) pay from about 20 wedges an edge on
@pytest.mark.parametrize("nu,nv,m,gamma,masks", [(400_000, 400_000, 600_000, 0, False),
                                                 (300_000, 300_000, 300_000, 2.5, False),
                                                 (100_000, 20_000, 1_000_000, 2.1, True)])
def test_masks_where_they_pay(R, nu, nv, m, gamma, masks):
    import torch
    eu, ev = synth.chung_lu(nu, nv, m, gamma, gamma, 2) if gamma else synth.er(nu, nv, m, 2)
    g = R.Graph(eu, ev, nu, nv)
    cu, cv = oracle.count_vp(eu, ev, nu, nv)
    lib, pool, v = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(), ctypes.c_uint64(0)
    assert lib.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    high = []
    for limit in (-1, 0):
        R.receipt_optional_memory(limit)
        torch.cuda.synchronize()
        v.value = 0
        assert lib.cuMemPoolSetAttribute(pool, 8, ctypes.byref(v)) == 0  # most bytes used
        gu, gv = g.count_butterflies()
        R.receipt_optional_memory(-1)
        torch.cuda.synchronize()
        assert lib.cuMemPoolGetAttribute(pool, 8, ctypes.byref(v)) == 0
        high.append(v.value)
        assert np.array_equal(R.as_u64(gu), cu) and np.array_equal(R.as_u64(gv), cv)
    if not masks:
        assert high[0] == high[1]
    else:
        assert high[0] != high[1]
