"""Tile rows that a context reports can be passed back, and the set-up's choice can be returned to after
another one has been tried; the apply keeps its bits."""
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


# FP64 sets of small blocks, where the tuner takes 16 rows, one below its 64 MB (32 rows), and three
# levels (one choice per level)
@pytest.mark.parametrize("m,parts,groups", [((11, 9, 13), (2, 2, 3), None), ((9, 6, 7), (3, 2, 2), None),
                                            ((3, 2, 2), (1, 1, 1), None), ((12, 8, 8), (4, 2, 2), ((2, 2, 2),))])
def test_reported_rows_are_accepted(lib, m, parts, groups):
    p = I.box_problem(*m, parts, groups=groups, levels=3 if groups else 2, form="symmetric", uk_seed=3, lam=1.0,
                      n=0.5, nu_inf=1e-2)
    ctx = lib.Context(p)
    nl = ctx.sizes.levels - 1

    def rows_now():
        s = lib.gdsw_sizes_info()
        lib.load().gdsw_sizes(ctx.h, C.byref(s))
        return list(s.tile_rows)[:nl]

    r = torch.from_numpy(np.random.default_rng(1).standard_normal(ctx.n)).cuda()
    z, ref = torch.empty_like(r), torch.empty_like(r)
    ctx.gdsw_apply(r, ref)

    def same():
        ctx.gdsw_apply(r, z.fill_(float("nan")))
        torch.cuda.synchronize()
        return torch.equal(z, ref)

    chosen = rows_now()
    assert all(v in (16, 32, 64, 128) for v in chosen)
    for persistent in (False, True):
        for rows in sorted(set(chosen)):
            ctx.gdsw_set_local_sweep(persistent, 0, rows)
            assert rows_now() == [rows] * nl and same()
            ctx.gdsw_set_local_sweep(persistent, 0, -1)
            assert rows_now() == chosen and same()
        ctx.gdsw_set_local_sweep(persistent, 0, 128)
        assert rows_now() == [128] * nl and same()
        ctx.gdsw_set_local_sweep(persistent, 0, 0)
        assert rows_now() == [128] * nl and same()
        ctx.gdsw_set_local_sweep(persistent, 0, -1)
        assert rows_now() == chosen and same()
    for rows in (-2, 1, 8, 48, 256):
        with pytest.raises(lib.GdswError):
            ctx.gdsw_set_local_sweep(False, 0, rows)
    assert rows_now() == chosen and same()
    ctx.close()
