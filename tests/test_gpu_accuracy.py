"""How near the fixed-point kernels of the assembly come to the exact result,
where FP64 arithmetic itself would be near: the tolerances are those of the
kernels' own rounding."""
import itertools
import os

import numpy as np
import pytest

import lattice_inputs as LI
from oracle import rom as orom

pytestmark = pytest.mark.gpu
romb = pytest.importorskip("paper_2604_09113_gb300")

U = 2.0 ** -53


@pytest.mark.parametrize("r,n_r", [(1, 20), (2, 33), (6, 60), (6, 127), (10, 40)])
def test_theta_of_small_samples(r, n_r, tmp_path):
    """At the corners of the box every weight is exactly 0 or 1, so theta is one
    sample: rounded to 2^-57 of the largest sample of its coefficient (59 bits
    below four times that), and to FP64 (the sum, 1 - rho, their product).  The
    samples there are 2^-10 of the others."""
    g = np.random.default_rng(r + n_r)
    p, n_i = 3, 4 ** 4 * 36
    A = g.uniform(-1, 1, size=(n_r, r + 1, r + 1, r + 1, r + 1))
    ends = [0, r]
    for c in itertools.product(ends, repeat=4):
        A[(slice(None),) + c] *= 2.0 ** -10
    A[:, 1 if r > 1 else 0, 0, 0, 0] = 1.0
    R = orom.Rom(0, 0, p, 2, r, 0.125, 0.375, g.standard_normal(n_i), g.standard_normal((n_i, n_r)) / np.sqrt(n_i),
                 A.reshape(n_r, -1), np.arange(n_r))
    path = os.path.join(str(tmp_path), "m.rom")
    orom.write(R, path)
    lat = LI.lattice(4, 4, p, 1, seed=9, geometry="affine", mu_mode="uniform", mu_range=(0.13, 0.37))
    corners = np.array(list(itertools.product(ends, repeat=4)))   # thresholds 4, 3, 2, 1 of the grid order
    lat.mu = np.where(corners[:, ::-1] > 0, 0.375, 0.125)
    with romb.Context(0) as ctx:
        romb.romb_train_load(ctx.h, path)
        romb.romb_assemble(ctx.h, lat, romb.ROMB_FP64)
        th = romb.romb_read(ctx.h, "theta").reshape(lat.ncells, -1)[:, 1:]
    for c in range(lat.ncells):
        ref = (1 - lat.rho) * A[(slice(None),) + tuple(corners[c])]
        assert np.all(np.abs(th[c] - ref) <= 2.0 ** -57 * np.abs(A).reshape(n_r, -1).max(axis=1) + 3 * U * np.abs(ref)), c
