"""The robust inner problem within its 256 bytes of workspace: no device memory is taken for the
columns' common order, from one row to more rows than the launch has warps."""
import ctypes

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
afc = pytest.importorskip("paper_2605_14743_gb300")

USED_MEM_CURRENT, USED_MEM_HIGH = 7, 8   # CU_MEMPOOL_ATTR_USED_MEM_*


def _inner(counts, R, v, support_only, qstar):
    n = counts.shape[0]
    ch = afc.Chain()
    ch.n, ch.realizations, ch.alpha, ch.absorb_floor = n, R, 0.1, 1e-6
    T = torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
    Qs = torch.empty((n, n), dtype=torch.float64, device="cuda") if qstar else None
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    afc.afc_robust_inner(ch, counts, 0.05, 0.05, support_only, v, 0.3, T, Qs, ws,
                         torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return T.cpu().numpy(), None if Qs is None else Qs.cpu().numpy()


def _small(n, seed):
    rng = np.random.default_rng(seed)
    R = 5000
    c = rng.multinomial(R, rng.dirichlet(np.ones(n + 1)), size=n).astype(np.uint32)
    c[rng.random(c.shape) < 0.5] = 0
    c[:, n] += (R - c.sum(1)).astype(np.uint32)
    return c, R, rng.normal(size=n)


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


@pytest.mark.parametrize("n", [1, 2, 8, 9, 33, 90])
@pytest.mark.parametrize("support_only", [0, 1])
def test_small_problems(n, support_only):
    c, R, v = _small(n, n)
    Q, _ = O.assemble_q(c, R, 0.1)
    oT, oQ = O.robust_inner(Q, 0.05, 0.05, v, 0.3, bool(support_only))
    for qstar in (False, True):
        T, Qs = _inner(_cuda(c), R, torch.from_numpy(v).cuda(), support_only, qstar)
        assert np.allclose(T, oT, rtol=0, atol=1e-9)
        assert Qs is None or np.allclose(Qs, oQ, rtol=0, atol=1e-9)


def test_more_rows_than_warps():
    """10,001 rows that repeat 60 small ones, on 60 spread columns."""
    k, n = 60, 10001
    c, R, v = _small(k, 3)
    at = np.arange(k) * 160 + 5
    counts = torch.zeros((n, n + 1), dtype=torch.int32, device="cuda")
    rows = torch.arange(n, device="cuda") % k
    counts[:, torch.from_numpy(at).cuda()] = _cuda(c[:, :k])[rows]
    counts[:, n] = _cuda(c)[:, k][rows]
    vb = np.random.default_rng(1).normal(size=n)
    vb[at] = v
    Q, _ = O.assemble_q(c, R, 0.1)
    oT, _ = O.robust_inner(Q, 0.05, 0.05, v, 0.3, True)
    T, _ = _inner(counts, R, torch.from_numpy(vb).cuda(), 1, False)
    assert np.allclose(T, oT[np.arange(n) % k], rtol=0, atol=1e-9)


def test_no_device_memory_is_taken():
    cu = ctypes.CDLL("libcuda.so.1")
    c, R, v = _small(90, 1)
    ct, vt = _cuda(c), torch.from_numpy(v).cuda()
    _inner(ct, R, vt, 1, True)
    pool, high, now = ctypes.c_void_p(), ctypes.c_uint64(0), ctypes.c_uint64(0)
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    assert cu.cuMemPoolSetAttribute(pool, USED_MEM_HIGH, ctypes.byref(high)) == 0
    _inner(ct, R, vt, 1, True)
    assert cu.cuMemPoolGetAttribute(pool, USED_MEM_HIGH, ctypes.byref(high)) == 0
    assert cu.cuMemPoolGetAttribute(pool, USED_MEM_CURRENT, ctypes.byref(now)) == 0
    assert high.value == now.value
