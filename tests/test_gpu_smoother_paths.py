"""FP32 smoothing of the multigrid in both of its forms -- element by element, and from an FP32 copy of
the rows when the operator holds the Newton term -- against FP64 smoothing.

Tolerance: one sweep is a chain of eight residuals and patch solves in FP32 (eps 6e-8) whose
contributions of up to 402 terms partly cancel; the oracle's FP32 emulation and the assembled form both
stay below 4e-7 relative on these data, a wrong or missing term is above 1e-3: 2e-6."""
import ctypes as C

import numpy as np
import pytest

from paper_2606_01433_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_01433_gb300 import gdsw
    gdsw.load()
    return gdsw


def _smooth(g, seed):
    rng = np.random.default_rng(seed)
    b, x = (torch.from_numpy(rng.standard_normal(g.n)).cuda() for _ in range(2))
    z = torch.zeros_like(b)
    g.gdsw_mg_smooth(0, b, x, 1)
    g.gdsw_mg_smooth(0, b, z, 2)
    torch.cuda.synchronize()
    return x.cpu().numpy(), z.cpu().numpy()


def _close(a, b):
    for u, v in zip(a, b):
        assert np.linalg.norm(u - v) <= 2e-6 * np.linalg.norm(v)


@pytest.mark.parametrize("m", [4, 6, 10, 16])
@pytest.mark.parametrize("carreau", [True, False])
def test_element_smoothing(lib, m, carreau):
    """8, 27, 125 and 512 patches per colour (the next grid of a 2-element one would be singular); both forms of the viscous term."""
    out = {}
    for sm in ("fp64", "fp32"):
        probs = I.mg_hierarchy(m, 2, parts=(1, 1, 1), groups=(), levels=2, seed=m, carreau=carreau)
        g = lib.Multigrid(probs, smoother=sm, symmetric=True)
        out[sm] = _smooth(g, 3)
        again = _smooth(g, 3)
        assert all(np.array_equal(u, v) for u, v in zip(out[sm], again))
        g.close()
    _close(out["fp32"], out["fp64"])


def test_jacobian_smoothing(lib):
    """After a Newton step the finest context holds the Jacobian: the smoother of a multigrid created
    then takes its FP32 values."""
    probs = I.mg_hierarchy(8, 2, parts=(2, 2, 2), groups=(), levels=2, seed=5, n=0.4, nu_inf=1e-2)
    g = lib.Multigrid(probs, smoother="fp32", tol=1e-8, symmetric=True)
    x = torch.zeros(g.n, dtype=torch.float64, device="cuda")
    g.grids[0].gdsw_picard_update(x)
    g.grids[0].newton_step(x)
    out = {}
    for sm in ("fp64", "fp32"):
        g.lib.gdsw_mg_destroy(g.h)
        g.h = None
        arr = (C.c_void_p * len(g.grids))(*[c.h.value for c in g.grids])
        o = lib.gdsw_mg_options(1.0, 2, 2, lib.PREC[sm], 1)
        h = C.c_void_p()
        assert g.lib.gdsw_mg_create(arr, len(g.grids), C.byref(o), C.byref(h)) == lib.GDSW_OK
        g.h = h
        out[sm] = _smooth(g, 4)
    _close(out["fp32"], out["fp64"])
    g.close()
