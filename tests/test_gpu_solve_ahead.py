"""Solves that stop at every kind of place while the next iteration is already queued: at an iteration
limit, at the end of a restart cycle, at a loose and at a tight tolerance, on a small system and on one
that takes many cycles.  The solution has to be the one of exactly the counted iterations: its
true residual equals the estimate of the last of them.

Tolerance: estimate and true residual of an FGMRES cycle differ by the loss of orthogonality of twice
orthogonalised vectors, 1e-14 of ||b||; residuals here are above 1e-10 of it: 1e-3 of the estimate."""
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


@pytest.mark.parametrize("max_it", [1, 2, 3, 4, 7, 12, 200])
@pytest.mark.parametrize("restart", [3, 7, 100])
@pytest.mark.parametrize("tol", [1e-2, 1e-9])
def test_counted_iterations(lib, max_it, restart, tol):
    p = I.box_problem(6, 5, 4, (2, 2, 1), levels=2, form="symmetric", uk_seed=3, lam=1.0, n=0.5, nu_inf=1e-2)
    ctx = lib.Context(p, precision=("fp32",) * 3, phi_precision="fp32", tol=tol, max_it=max_it, restart=restart)
    b = torch.from_numpy(np.random.default_rng(5).standard_normal(ctx.n)).cuda()
    x, ax = torch.zeros_like(b), torch.zeros_like(b)
    info = ctx.gdsw_solve(b, x)
    ctx.gdsw_spmv(x, ax)
    true = float(torch.linalg.norm(b - ax) / torch.linalg.norm(b))
    assert info.iterations <= max_it
    assert info.iterations == max_it or info.relres <= tol
    assert abs(true - info.relres) <= 1e-10 * (1 + true)
    assert abs(info.est_relres - info.relres) <= 1e-3 * info.est_relres
    ctx.close()


def test_many_contexts(lib):
    """More contexts alive at once than the shared page has estimate pairs (256); pairs given back are
    used again."""
    p = I.box_problem(3, 3, 3, (1, 1, 1), levels=2, form="symmetric", uk_seed=3, lam=1.0, n=0.5, nu_inf=1e-2)
    ref = None
    for count in (258, 2):
        ctxs = [lib.Context(p, tol=1e-10) for _ in range(count)]
        b = torch.from_numpy(np.random.default_rng(5).standard_normal(ctxs[0].n)).cuda()
        for c in ctxs:
            x = torch.zeros_like(b)
            assert c.gdsw_solve(b, x).relres <= 1e-10
            ref = x if ref is None else ref
            assert torch.equal(x, ref)
        for c in ctxs:
            c.close()
