"""The Arnoldi launches where their shapes change: a partly filled CTA, one CTA, one group of
CTAs, several groups, several rows per warp, more basis vectors than are staged at a time (64), and a
restart.  A solve must reach its true residual, be the same bit for bit when repeated, and agree
with a dense solution on the small sizes.

Tolerance of the dense comparison: the solve stops at 1e-12; the condition numbers of these systems
are 2e4 to 1e5, so 1e-7."""
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


def _solve(lib, p, seed, **kw):
    ctx = lib.Context(p, **kw)
    b = torch.from_numpy(np.random.default_rng(seed).standard_normal(ctx.n)).cuda()
    x, x2 = torch.zeros_like(b), torch.zeros_like(b)
    info = ctx.gdsw_solve(b, x)
    ctx.gdsw_solve(b, x2)
    r = torch.empty_like(b)
    ctx.gdsw_residual(b, x, r)
    torch.cuda.synchronize()
    assert info.status == 0
    assert torch.equal(x, x2)
    relres = float(torch.linalg.norm(r) / torch.linalg.norm(b))
    assert relres <= 1.01 * kw["tol"] and abs(relres - info.relres) <= 1e-14
    return ctx, b, x, info


@pytest.mark.parametrize("m,parts", [((2, 2, 2), (1, 1, 1)), ((2, 2, 3), (2, 1, 1)), ((3, 3, 3), (2, 2, 2)),
                                     ((5, 4, 6), (2, 2, 2))])
def test_small_solves_match_dense(lib, m, parts):
    p = I.box_problem(*m, parts, levels=2, form="symmetric", uk_seed=3, lam=1.0, n=0.5, nu_inf=1e-2)
    ctx, b, x, _ = _solve(lib, p, 1, tol=1e-12)
    A = ctx.gdsw_matrix_csr().toarray()
    ref = np.linalg.solve(A, b.cpu().numpy())
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-7 * np.linalg.norm(ref)
    ctx.close()


@pytest.mark.parametrize("m,parts,restart", [((12, 12, 12), (4, 4, 4), 100), ((20, 20, 20), (5, 5, 5), 100),
                                             ((10, 9, 11), (3, 3, 3), 20)])
def test_solves_over_the_launch_shapes(lib, m, parts, restart):
    """40 thousand dofs (two groups of CTAs), 185 thousand (two rows per warp), and restarts; plain
    weighting, which takes more iterations, so that more than 64 basis vectors occur."""
    p = I.box_problem(*m, parts, levels=2, form="symmetric", uk_seed=3, lam=1.0, n=0.4, nu_inf=1e-3)
    ctx, _, _, info = _solve(lib, p, 2, tol=1e-12, precision=("fp32",) * 3, phi_precision="fp32", restart=restart,
                             weighting="plain")
    assert info.iterations > (64 if restart == 100 else restart)
    ctx.close()
