"""The batched Gauss-Jordan inverse over the forms of its panel: one CTA of 64, 128 and 256 threads,
clusters of 2 to 8 CTAs, two rows per thread, more rows than a cluster holds, and batches of
different sizes.  With slab_elems = 0 a part's matrix is one dense block, and with one part the local
solve is A^{-1} itself.

Tolerance (FP64): the residual of a computed inverse is at most about n eps cond(A) relative to the
right-hand side; n <= 6e3, eps = 1.1e-16, cond <= 2e5 (the meshes' systems measure 2e4 to 1e5): 1.4e-7,
and the growth of partial pivoting is far from its bound; 1e-8 holds with a margin in practice and
is a hundred times below what a lost digit of single precision would leave.  FP32 (eps 6e-8) is only
a preconditioner: FGMRES must reach 1e-10 within 12 steps, three digits per step being the least
that an inverse of that accuracy gives."""
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


# n = 72, 135, 297, 514, 982, 1662, 2520, 3858, 5540 rows in the first panel
MESHES = [(1, 2, 2), (2, 2, 2), (2, 2, 4), (3, 3, 3), (3, 4, 4), (4, 4, 5), (5, 4, 6), (6, 5, 6), (6, 6, 7)]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("m", MESHES)
def test_one_dense_block(lib, m, prec):
    p = I.box_problem(*m, (1, 1, 1), levels=2, form="symmetric", uk_seed=3, lam=1.0, n=0.5, nu_inf=1e-2)
    ctx = lib.Context(p, precision=(prec,) * 3, phi_precision=prec, slab_elems=0, tol=1e-10)
    r = torch.from_numpy(np.random.default_rng(3).standard_normal(ctx.n)).cuda()
    z, y = torch.zeros_like(r), torch.zeros_like(r)
    if prec == "fp64":
        ctx.gdsw_apply_local(0, r, z)
        ctx.gdsw_spmv(z, y)
        assert float(torch.linalg.norm(y - r) / torch.linalg.norm(r)) <= 1e-8
    else:
        info = ctx.gdsw_solve(r, z)
        assert info.status == 0 and info.iterations <= 12
    ctx.close()


def test_ragged_batch(lib):
    """Parts of different sizes in one batch (a die cut by bisection): the two-level solve converges
    as with exact local solvers."""
    p = I.die(16, 16, 32, nparts=16, per_group=4, levels=2)
    its = []
    for prec in ("fp64", "fp32"):
        ctx = lib.Context(p, precision=(prec,) * 3, phi_precision=prec, tol=1e-10)
        b = torch.zeros(ctx.n, dtype=torch.float64, device="cuda")
        ctx.gdsw_rhs_lift(b)
        x = torch.zeros_like(b)
        info = ctx.gdsw_solve(b, x)
        assert info.status == 0
        its.append(info.iterations)
        ctx.close()
    assert abs(its[0] - its[1]) <= 2
