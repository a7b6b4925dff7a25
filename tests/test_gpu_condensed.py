"""Local solves of sets whose factors are large enough for the condensed form (mid planes eliminated
first), against FP64 solves with slabs two elements thick, which are never condensed: the same
A_i^{-1}, factorised in another way.

Tolerances: FP64 5e-16 and FP32 6e-8 rounding on blocks of up to 8000 dofs whose condition stays below
1e5: 1e-8 and 1e-2 for a vector A x (whose solution x the solve returns); BF16 entries carry 2^-9
each: 2e-2 of a solve of random data.  A missing coupling is an error of the order of one."""
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


def _box(m, parts, pressure):
    return I.box_problem(*m, parts, levels=2, form="symmetric", uk_seed=3, lam=1.0, n=0.5, nu_inf=1e-2,
                         pressure=pressure)


def _solves(lib, p, prec, slab_elems=1):
    ctx = lib.Context(p, precision=(prec,) * 3, phi_precision="fp64" if prec == "fp64" else "fp32",
                      slab_elems=slab_elems)
    r = torch.from_numpy(np.random.default_rng(1).standard_normal(ctx.n)).cuda()
    ax = torch.zeros_like(r)
    ctx.gdsw_spmv(r, ax)
    out = []
    for persistent in (False, True):
        for rows in (0, 32, 128):
            ctx.gdsw_set_local_sweep(persistent, 0, rows)
            zs = [torch.full_like(r, float("nan")) for _ in range(2)]
            ctx.gdsw_apply_local(0, r, zs[0])
            ctx.gdsw_apply_local(0, ax, zs[1])
            torch.cuda.synchronize()
            assert not out or all(torch.equal(u, v) for u, v in zip(out, zs))
            out = zs
    entries = ctx.sizes.factor_entries[0]
    ctx.close()
    return out, entries


def _err(u, v):
    return float(torch.linalg.norm(u - v) / torch.linalg.norm(v))


@pytest.mark.parametrize("m,parts,pressure", [((19, 13, 13), (2, 1, 1), "q1"), ((12, 12, 17), (1, 1, 1), "p1disc")])
def test_condensed_matches_thick_slabs(lib, m, parts, pressure):
    p = _box(m, parts, pressure)
    ref, thick = _solves(lib, p, "fp64", slab_elems=2)
    for prec, tol in (("fp64", 1e-8), ("fp32", 1e-2)):
        z, entries = _solves(lib, p, prec)
        assert entries < 0.5 * thick          # plain slabs of one element hold more than half of that
        assert _err(z[0], ref[0]) <= tol and _err(z[1], ref[1]) <= tol


def test_condensed_irregular(lib):
    """Obstacles: planes with gaps, parts of different shape, mid planes without a plane below."""
    p = I.channel(20, parts=(2, 2, 2), groups=(), levels=2, seed=2, n=0.5)
    ref, thick = _solves(lib, p, "fp64", slab_elems=2)
    z, entries = _solves(lib, p, "fp32")
    assert entries < 0.5 * thick
    assert _err(z[0], ref[0]) <= 1e-2 and _err(z[1], ref[1]) <= 1e-2
    zb, _ = _solves(lib, p, "bf16")
    assert _err(zb[0], ref[0]) <= 2e-2
