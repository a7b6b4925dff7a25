"""An iteration that was queued before its predecessor turned out to have converged is dropped: the profile
counts it, the solution does not hold it.  The tolerance is laid between an estimate that falls faster than
the solver foresees and what it foresees for that iteration."""
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


@pytest.mark.parametrize("weighting", ["pou", "plain"])
@pytest.mark.parametrize("m,parts", [((2, 2, 2), (2, 2, 2)), ((2, 2, 2), (2, 1, 1)), ((3, 2, 1), (3, 2, 1))])
def test_dropped_iteration(lib, m, parts, weighting):
    p = I.box_problem(*m, parts, levels=2, form="symmetric", uk_seed=3, lam=1.0, n=0.4, nu_inf=1e-3)

    def context(**kw):
        return lib.Context(p, precision=("fp32",) * 3, phi_precision="fp32", weighting=weighting, **kw)

    def solve(ctx, x):
        info = ctx.gdsw_solve(b, x)
        torch.cuda.synchronize()
        return info

    b, h = None, []
    for j in range(1, 9):  # estimates of the first iterations (at a limit nothing is queued ahead of it)
        ctx = context(tol=1e-30, max_it=j)
        if b is None:
            b = torch.zeros(ctx.n, dtype=torch.float64, device="cuda")
            ctx.gdsw_rhs_lift(b)
        h.append(solve(ctx, torch.zeros_like(b)).est_relres)
        ctx.close()
    foreseen = [np.inf] * 3 + [0.3 * h[k - 1] * min(1.0, h[k - 1] / h[k - 2]) for k in range(3, 8)]
    k = next(k for k in range(3, 8) if h[k] < 0.9 * foreseen[k])
    tol = float(np.sqrt(h[k] * foreseen[k]))
    # the solution without the queued iteration: k + 1 iterations, then what the true residual asks for
    y = torch.zeros_like(b)
    ctx = context(tol=tol, max_it=k + 1)
    first = solve(ctx, y)
    ctx.close()
    assert first.iterations == k + 1 and first.est_relres <= tol
    rest = 0
    if first.relres > tol:
        ctx = context(tol=tol)
        rest = solve(ctx, y).iterations
        ctx.close()
    ctx = context(tol=tol)
    ctx.gdsw_profile_enable(1)
    for _ in range(2):  # again with what the dropped iteration left in the workspace
        x = torch.zeros_like(b)
        ctx.gdsw_profile_reset()
        info = solve(ctx, x)
        assert info.status == 0 and info.relres <= tol and info.iterations == k + 1 + rest
        assert ctx.gdsw_profile_read()["arnoldi"]["calls"] > info.iterations
        assert torch.equal(x, y)
    ctx.close()
