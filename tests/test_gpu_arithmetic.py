"""romb_set_fp64_arithmetic: what it reaches, and that it stays the caller's."""
import numpy as np
import pytest

import lattice_inputs as LI

from romb_testutil import small_rom, unpack_upper

pytestmark = pytest.mark.gpu
romb = pytest.importorskip("paper_2604_09113_gb300")
torch = pytest.importorskip("torch")
from paper_2604_09113_gb300.autograd import compliance  # noqa: E402


def _lat(p, nx=4, ny=3):
    return LI.lattice(nx, ny, p, 2, seed=41, mu_mode="uniform", mu_range=(0.22, 0.36), rho=5e-4)


def _k(ctx, lat):
    romb.romb_assemble(ctx.h, lat, romb.ROMB_FP64)
    return romb.romb_read(ctx.h, "K")


@pytest.mark.parametrize("precision", ["ROMB_FP64", "ROMB_FP32_SPLIT"])
@pytest.mark.parametrize("pipe", [False, True])
def test_a_gradient_leaves_the_choice(pipe, precision):
    """The matrices of a plain FP64 assembly are the same, bit by bit, before and
    after a compliance with its gradient on the same context."""
    lat = _lat(4)
    _, path = small_rom(0, 4, 0.18, 0.40, 20, 12, 1)
    with romb.Context(0) as ctx:
        romb.romb_train_load(ctx.h, path)
        other = _k(ctx, lat)
        romb.romb_set_fp64_arithmetic(ctx.h, pipe)
        before = _k(ctx, lat)
        assert np.array_equal(before, other) != pipe   # the choice shows in K
        ctrl = torch.tensor(lat.ctrl, requires_grad=True)
        mu = torch.tensor(lat.mu, requires_grad=True)
        compliance(ctx, lat, ctrl, mu, getattr(romb, precision), rtol=1e-8).backward()
        assert np.array_equal(_k(ctx, lat), before)
