"""Device memory of the 3-RDM: twice n^2 vectors of the determinant length, of
which one n^2 counts at least 1 GiB, and about 1 GiB for the operands of the
products under way, whatever the size; and the same values over several
ranges of K as the oracle gives over one."""
import ctypes

import numpy as np
import pytest

from gbd_synth import make_integrals

pytestmark = pytest.mark.gpu

USED_HIGH = 8   # CU_MEMPOOL_ATTR_USED_MEM_HIGH


@pytest.fixture(scope="module")
def G():
    from paper_2609_09990_gb300 import build, gbdmrg
    build.build()
    return gbdmrg


def pool_high(reset):
    """High-water mark of the default memory pool of device 0 since the last reset, bytes."""
    cu = ctypes.CDLL("libcuda.so.1")
    pool, v = ctypes.c_void_p(), ctypes.c_uint64(0)
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    f = cu.cuMemPoolSetAttribute if reset else cu.cuMemPoolGetAttribute
    assert f(pool, USED_HIGH, ctypes.byref(v)) == 0
    return v.value


@pytest.mark.parametrize("n,M", [(11, 24), (12, 16)])
def test_peak(G, n, M):
    h, chol = make_integrals(n, 2 * n, 3)
    ne = n - n % 2
    ctx = G.Context(0)
    ctx.solve(h, chol, ne, 0, [M], [1e-3], seed=3)
    from math import comb
    ndet = comb(n, ne // 2) ** 2
    pool_high(True)
    g3 = ctx.rdm3(n)
    peak = pool_high(False)
    g1, g2 = ctx.rdms(n)
    ctx.close()
    vectors = 8 * n * n * ndet
    # vectors, batch, digits, and 0.4 GiB for partial sums, lists and the state
    assert peak <= vectors + max(vectors, 1 << 30) + 1.4 * 2 ** 30, peak / 2 ** 30
    scale = np.abs(g3).max()
    assert np.abs(np.einsum("pqrsuu->pqrs", g3) - (ne - 2) * g2).max() <= 1e-10 * scale
    assert np.abs(np.einsum("ppqrst->qrst", g3) - (ne - 2) * g2).max() <= 1e-10 * scale
    assert np.abs(g3 - g3.transpose(1, 0, 3, 2, 5, 4)).max() <= 1e-11 * scale
