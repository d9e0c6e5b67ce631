"""The digit tiles of the FP64 form take only memory that nothing else needs:
whatever a budget admits with the contraction on the FP64 pipe, which has no
tiles, it also admits in the default arithmetic."""
import numpy as np
import pytest

import lattice_inputs as LI

from romb_testutil import small_rom

pytestmark = pytest.mark.gpu
romb = pytest.importorskip("paper_2604_09113_gb300")


def _lattices(p):
    out = []
    for nx, ny in ((5, 3), (9, 6)):
        lat = LI.lattice(nx, ny, p, 2, seed=3, mu_mode="uniform", mu_range=(0.2, 0.38))
        lat.family = (np.arange(lat.ncells) % 3 == 1).astype(np.int32)
        out.append(lat)
    return out


def _steps(budget, pipe, paths, lats):
    """Two lattices, the second larger: assembled, factorised and solved with two
    load sets twice, then a gradient."""
    out = []
    with romb.Context(0, mem_budget_bytes=budget) as ctx:
        for path in paths:
            romb.romb_train_load(ctx.h, path)
        romb.romb_set_fp64_arithmetic(ctx.h, pipe)
        for lat in lats:
            nodes = (lat.p * lat.nx + 1) * (lat.p * lat.ny + 1)
            for _ in range(2):
                romb.romb_assemble(ctx.h, lat, romb.ROMB_FP64)
                romb.romb_factor(ctx.h)
                u, _, _ = romb.romb_bddc_solve(ctx.h, nodes, nrhs=2, traction_sets=LI.traction_sets(2, 5), rtol=1e-12,
                                               maxit=500)
                out.append(u.copy())
            romb.romb_bddc_solve(ctx.h, nodes, rtol=1e-12, maxit=500)
            out.append(romb.romb_compliance_grad(ctx.h, len(lat.ctrl), lat.ncells)[3])
    return out


def _fits(budget, *args):
    try:
        _steps(budget, *args)
    except romb.RombError as e:
        assert "memory" in str(e), e
        return False
    return True


def test_tiles_leave_every_budget_as_it_was():
    p = 4
    paths = [small_rom(f, p, 0.18, 0.40, 20, 12, 1)[1] for f in (0, 1)]
    lats = _lattices(p)
    ref = _steps(0, False, paths, lats)
    lo, hi = 1 << 16, 1 << 28   # the least budget of the work without tiles, to 4 KB
    assert _fits(hi, True, paths, lats) and not _fits(lo, True, paths, lats)
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if _fits(mid, True, paths, lats) else (mid, hi)
    tiles = 325 * 8 * 40 * 2 * 16   # of one model: pairs, digits, rows, bytes, K padded
    for extra in (0, tiles // 2, tiles + tiles // 2, 2 * tiles + 65536):
        got = _steps(hi + extra, False, paths, lats)
        for a, b in zip(got, ref):
            assert np.abs(a - b).max() <= 1e-8 * np.abs(b).max(), extra
