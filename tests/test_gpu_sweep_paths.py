"""Local solves with every tile shape, as step launches and as the persistent launch: the same bits in
each storage precision (a row's dot product and its sum over the warp have one order whatever the
tile), and the solve's accuracy against the assembled operator (one part: the local solve is A^{-1})."""
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


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("m,parts", [((3, 2, 2), (1, 1, 1)), ((9, 6, 7), (3, 2, 2)), ((14, 13, 12), (2, 2, 2))])
def test_tile_shapes_agree(lib, prec, m, parts):
    p = I.box_problem(*m, parts, levels=2, form="symmetric", uk_seed=3, lam=1.0, n=0.5, nu_inf=1e-2)
    ctx = lib.Context(p, precision=(prec,) * 3, phi_precision="fp64" if prec == "fp64" else "fp32")
    r = torch.from_numpy(np.random.default_rng(1).standard_normal(ctx.n)).cuda()
    ref = None
    for persistent in (False, True):
        # rows = 0: the tiles that the set-up chose, of 16 rows where the matrices are small
        for rows in (0, 32, 64, 128):
            ctx.gdsw_set_local_sweep(persistent, 0, rows)
            z = torch.full_like(r, float("nan"))
            ctx.gdsw_apply_local(0, r, z)
            torch.cuda.synchronize()
            assert bool(torch.isfinite(z).all())
            ref = z if ref is None else ref
            assert torch.equal(z, ref), (persistent, rows)
    if prec == "fp64" and parts == (1, 1, 1):
        y = torch.zeros_like(r)
        ctx.gdsw_spmv(ref, y)
        assert float(torch.linalg.norm(y - r) / torch.linalg.norm(r)) <= 1e-9
    with pytest.raises(lib.GdswError):
        ctx.gdsw_set_local_sweep(False, 0, 16)
    ctx.close()
