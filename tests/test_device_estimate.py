"""The device memory that the analysis reports, by which the solve server admits requests: a request that
fitted a budget keeps fitting it.  The bounds are the reports of the assembly without a workspace of its
own, which the element blocks (29 KB per element) must not add to from 8^3 elements on."""
import pytest

from paper_2606_01433_gb300 import inputs as I


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_01433_gb300 import gdsw
    gdsw.load()
    return gdsw


def _box(m, parts):
    return I.box_problem(*m, parts, levels=2, form="symmetric", uk_seed=3, lam=1.0, n=0.5, nu_inf=1e-2)


@pytest.mark.parametrize("prob,prec,bound", [
    (lambda: I.carreau_cube(8, 0.5, 1e-3, seed=1), "fp32", 164205176),
    (lambda: I.carreau_cube(20, 0.5, 1e-3, seed=1), "fp32", 4514514336),
    (lambda: _box((8, 8, 8), (2, 2, 2)), "fp64", 274017848),
    (lambda: _box((8, 8, 8), (2, 2, 2)), "bf16", 137013304),
    (lambda: _box((8, 8, 8), (4, 4, 4)), "fp32", 159913784),
    (lambda: _box((14, 13, 12), (2, 2, 2)), "fp32", 1194622700),
    (lambda: _box((14, 13, 12), (2, 2, 2)), "bf16", 961072396),
    (lambda: _box((16, 16, 16), (8, 8, 8)), "bf16", 1429497284),
    (lambda: _box((20, 20, 20), (4, 4, 4)), "bf16", 3629469728),
])
def test_estimate_does_not_grow(lib, prob, prec, bound):
    ctx = lib.Context(prob(), analyze_only=True, precision=(prec,) * 3,
                       phi_precision="fp64" if prec == "fp64" else "fp32")
    assert 0 < ctx.sizes.device_bytes <= bound
    ctx.close()
