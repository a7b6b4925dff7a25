"""The operator kernels at the sizes where their launch shapes change: one element (half an element
CTA), an odd count, more elements than the assembly workspace holds (two chunks), both forms and
both pressure elements, against the FP64 oracle.

Tolerance: an entry is the sum of at most 8 x 27 products of five factors, each rounded a few
times, and the products' magnitudes sum to a few times the largest entry: 216 x 4 x 1.1e-16 of it,
rounded up to 1e-13.  Vectors (lifting, products) add at most 8 such terms per row in another
order: the same bound on the relative 2-norm.
"""
import numpy as np
import pytest

from paper_2606_01433_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-13


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_01433_gb300 import gdsw
    gdsw.load()
    return gdsw


def _problem(m, form, pressure):
    kw = dict(uk_seed=3, lam=1.0, n=0.5, nu_inf=1e-3) if form == "symmetric" else {}
    return I.box_problem(*m, (1, 1, 1), levels=2, form=form, pressure=pressure, **kw)


@pytest.mark.parametrize("form", ["symmetric", "gradient"])
@pytest.mark.parametrize("m,pressure", [((1, 1, 1), "q1"), ((1, 1, 2), "p1disc"), ((3, 3, 3), "q1"),
                                        ((5, 3, 2), "p1disc"), ((21, 21, 21), "q1")])
def test_assembled_operator(lib, m, pressure, form):
    from oracle import fem
    p = _problem(m, form, pressure)
    S = fem.assemble(p)
    ctx = lib.Context(p, levels=1)
    A, O = ctx.gdsw_matrix_csr(), S["A"]
    assert A.shape == O.shape
    scale = abs(O).max() if O.nnz else 1.0
    assert abs(A - O).max() <= TOL * scale
    # assembled again in place: the same numbers bit for bit
    ctx.gdsw_reassemble()
    assert np.array_equal(ctx.gdsw_matrix_csr().data, A.data)
    ctx.close()


@pytest.mark.parametrize("form", ["symmetric", "gradient"])
@pytest.mark.parametrize("m,pressure", [((1, 1, 2), "q1"), ((3, 3, 3), "p1disc"), ((5, 3, 2), "q1"), ((9, 4, 7), "p1disc")])
def test_viscosity_and_lifting(lib, m, pressure, form):
    """Gauss-point viscosity and lifted right-hand side: element counts around the eight elements of
    a viscosity CTA and the four of a lifting CTA; a Dirichlet datum on wall and inflow nodes."""
    from oracle import fem
    p = _problem(m, form, pressure)
    rng = np.random.default_rng(5)
    dirichlet = np.isin(p.tags, (I.TAG_WALL, I.TAG_INFLOW))
    p.g[dirichlet & (rng.random(p.n_nodes) < 0.4)] = rng.standard_normal(3)
    p.g[~dirichlet] = 7.0   # not a datum: must not be read
    S = fem.assemble(p)
    ctx = lib.Context(p, levels=1)
    nu = ctx.gdsw_viscosity_values()
    assert np.linalg.norm(nu - S["nu_q"]) <= TOL * np.linalg.norm(S["nu_q"])
    b = torch.full((ctx.n,), float("nan"), dtype=torch.float64, device="cuda")
    ctx.gdsw_rhs_lift(b)
    bo = fem.lifted_rhs(S)
    torch.cuda.synchronize()
    assert np.linalg.norm(b.cpu().numpy() - bo) <= TOL * max(np.linalg.norm(bo), 1e-300)
    ctx.close()


@pytest.mark.parametrize("m,pressure", [((1, 1, 1), "q1"), ((1, 2, 1), "p1disc"), ((8, 8, 8), "q1"), ((13, 12, 11), "q1"),
                                        ((13, 12, 13), "p1disc"), ((18, 19, 17), "q1")])
def test_products(lib, m, pressure):
    """y = A x and b - A x in every form of the product: slices of 8 rows with four and two warps,
    slices of 32 rows, and a partly filled last slice, against the assembled matrix.  A row has up
    to 375 + 27 terms: 402 x 1.1e-16, on the norms of |A| |x|."""
    p = _problem(m, "symmetric", pressure)
    ctx = lib.Context(p, levels=1)
    A = ctx.gdsw_matrix_csr()
    rng = np.random.default_rng(7)
    x, b = rng.standard_normal(ctx.n), rng.standard_normal(ctx.n)
    xd, bd = torch.from_numpy(x).cuda(), torch.from_numpy(b).cuda()
    y = torch.full_like(xd, float("nan"))
    r = torch.full_like(xd, float("nan"))
    ctx.gdsw_spmv(xd, y)
    ctx.gdsw_residual(bd, xd, r)
    torch.cuda.synchronize()
    bound = 402 * 1.1e-16 * (abs(A) @ abs(x) + abs(b))
    assert np.all(abs(y.cpu().numpy() - A @ x) <= bound)
    assert np.all(abs(r.cpu().numpy() - (b - A @ x)) <= bound)
    ctx.close()
