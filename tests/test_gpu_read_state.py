"""romb_read between romb_assemble and romb_factor: the fields of the last
factorisation are still its own (the assembly's scratch memory is not theirs),
and a new context has none of them in use."""
import numpy as np
import pytest

import lattice_inputs as LI

from romb_testutil import small_rom

pytestmark = pytest.mark.gpu
romb = pytest.importorskip("paper_2604_09113_gb300")

FIELDS = ("S", "psi", "sc_local", "D", "fine")


@pytest.mark.parametrize("p", [3, 4])
@pytest.mark.parametrize("form", ["ROMB_FP64", "ROMB_FP32_SPLIT", "ROMB_BF16_SPLIT"])
def test_assembly_leaves_the_last_factorisation(p, form):
    _, path = small_rom(0, p, 0.18, 0.40, 20, 12, 1)
    lat = LI.lattice(5, 3, p, 2, seed=3, mu_mode="uniform", mu_range=(0.2, 0.38))
    other = LI.lattice(5, 3, p, 2, seed=4, mu_mode="uniform", mu_range=(0.2, 0.38))
    with romb.Context(0) as ctx:
        romb.romb_train_load(ctx.h, path)
        romb.romb_assemble(ctx.h, lat, getattr(romb, form))
        romb.romb_factor(ctx.h)
        before = {f: romb.romb_read(ctx.h, f) for f in FIELDS}
        romb.romb_assemble(ctx.h, other, getattr(romb, form))
        for f in FIELDS:
            assert np.array_equal(romb.romb_read(ctx.h, f), before[f]), f
        other.mu[2, 1] = 0.9   # outside the box: the assembly is refused
        with pytest.raises(romb.RombError):
            romb.romb_assemble(ctx.h, other, getattr(romb, form))
        for f in FIELDS:
            assert np.array_equal(romb.romb_read(ctx.h, f), before[f]), f
