"""Contexts that come and go beside other work on the device: a set-up, a solve and the end of a context
wait for their own streams only."""
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


def test_no_wait_for_other_streams(lib):
    """A kernel of a second stream (2e9 cycles, about one second) is still running when a context's solve
    is done and when the process's only context has been destroyed, twice over."""
    p = I.carreau_cube(8, 0.5, 1e-3, seed=1)
    side, own = torch.cuda.Stream(), torch.cuda.Stream()
    ref = None
    for _ in range(3):
        with torch.cuda.stream(own):
            ctx = lib.Context(p, precision=("fp32",) * 3, phi_precision="fp32", tol=1e-10)
            b = torch.zeros(ctx.n, dtype=torch.float64, device="cuda")
            ctx.gdsw_rhs_lift(b)
            x = torch.zeros_like(b)
            ctx.gdsw_solve(b, x)   # whatever a process does once has been done
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(2_000_000_000)
            end = torch.cuda.Event()
            end.record()
        with torch.cuda.stream(own):
            x.zero_()
            info = ctx.gdsw_solve(b, x)
        solve_waited = end.query()
        ctx.close()
        close_waited = end.query()
        torch.cuda.synchronize()
        assert info.status == 0 and not solve_waited and not close_waited
        ref = x if ref is None else ref
        assert torch.equal(x, ref)


def test_many_contexts_solve_alike(lib):
    """Contexts alive at once, destroyed and made anew in another order: each keeps its own estimates."""
    p = I.carreau_cube(3, 0.5, 1e-3, seed=1)
    ctxs, ref = [], None
    for _ in range(24):
        ctxs.append(lib.Context(p, precision=("fp32",) * 3, phi_precision="fp32", tol=1e-10))
        if len(ctxs) == 16:
            for c in ctxs[::2]:
                c.close()
            ctxs = ctxs[1::2]
        for c in ctxs:
            b = torch.ones(c.n, dtype=torch.float64, device="cuda")
            x = torch.zeros_like(b)
            info = c.gdsw_solve(b, x)
            torch.cuda.synchronize()
            got = (x, info.iterations, info.est_relres)
            ref = got if ref is None else ref
            assert torch.equal(got[0], ref[0]) and got[1:] == ref[1:]
    for c in ctxs:
        c.close()
