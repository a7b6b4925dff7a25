"""Peak device memory of a set-up with many small parts, where the coarse operator's pieces are a large part
of it.  The bounds are the peaks with the interface products listed and summed as sorted segments; what
the device form accumulates in beside A_0 must stay below them."""
import ctypes as C
import gc

import pytest

from paper_2606_01433_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
USED_NOW, USED_HIGH = 7, 8  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, _HIGH


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_01433_gb300 import gdsw
    gdsw.load()
    return gdsw


@pytest.mark.parametrize("m,parts,group,prec,bound", [
    ((10, 10, 10), (5, 5, 5), (5, 5, 5), "fp32", 432.2e6),
    ((12, 12, 8), (6, 6, 4), (3, 3, 2), "fp32", 500.2e6),
    ((12, 12, 10), (6, 6, 5), (3, 3, 5), "bf16", 568.8e6),
    ((12, 12, 12), (6, 6, 6), (3, 3, 3), "fp32", 818.9e6),
])
def test_setup_peak(lib, m, parts, group, prec, bound):
    p = I.box_problem(*m, parts, groups=(group,), levels=3, form="symmetric", uk_seed=5, lam=1.0, n=0.6, nu_inf=1e-3)
    torch.zeros(1, device="cuda")
    gc.collect()  # contexts of other tests
    torch.cuda.synchronize()
    cu, pool, dev = C.CDLL("libcuda.so.1"), C.c_void_p(), torch.cuda.current_device()
    assert cu.cuDeviceGetDefaultMemPool(C.byref(pool), dev) == 0

    def read(attr):
        v = C.c_uint64(0)
        assert cu.cuMemPoolGetAttribute(pool, attr, C.byref(v)) == 0
        return v.value

    before = read(USED_NOW)
    assert cu.cuMemPoolSetAttribute(pool, USED_HIGH, C.byref(C.c_uint64(0))) == 0
    ctx = lib.Context(p, precision=(prec,) * 3, phi_precision="fp32", restart=20)
    torch.cuda.synchronize()
    peak = read(USED_HIGH) - before
    ctx.close()
    assert 0 < peak <= bound
