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


def _lagrange(nodes, x):
    n = len(nodes)
    v, d = np.ones(n, np.longdouble), np.zeros(n, np.longdouble)
    for i in range(n):
        for j in range(n):
            if j != i:
                d[i] = d[i] * (x - nodes[j]) + v[i]
                v[i] *= x - nodes[j]
        den = np.prod([nodes[i] - nodes[j] for j in range(n) if j != i])
        v[i], d[i] = v[i] / den, d[i] / den
    return v, d


def _chat(lat, c):
    """Chat at the nine interpolation nodes, [9][j1 j2][i1 i2], in extended precision."""
    from oracle import geometry as G
    P = G.cell_control_points(lat.ctrl, lat.nx, lat.m, c % lat.nx, c // lat.nx).astype(np.longdouble)
    lam, mu = (np.longdouble(v) for v in G.plane_stress_lame(lat.E, lat.nu))
    nodes = np.arange(lat.m + 1, dtype=np.longdouble) / lat.m
    out, I = [], np.eye(2, dtype=np.longdouble)
    for k in range(9):
        (v1, d1), (v2, d2) = _lagrange(nodes, k % 3 / 2), _lagrange(nodes, k // 3 / 2)
        J = np.stack([np.einsum("a,b,bac->c", d1, v2, P), np.einsum("a,b,bac->c", v1, d2, P)], axis=1)
        det = J[0, 0] * J[1, 1] - J[0, 1] * J[1, 0]
        g = np.array([[J[1, 1], -J[0, 1]], [-J[1, 0], J[0, 0]]]) / det
        C = lam * np.einsum("ji,lk->jlik", g, g)
        C += mu * (np.einsum("ik,jl->jlik", I, g @ g.T) + np.einsum("jk,li->jlik", g, g))
        out.append(det * C)
    return np.array(out)


@pytest.mark.parametrize("p,n_r,m", [(4, 20, 2), (6, 40, 3), (8, 80, 4)])
def test_contraction_keeps_rigid_translations(p, n_r, m, tmp_path):
    """What a rigid translation costs in K, by rows (K t) and as a whole (t K t):
    the digit products are no further from extended precision than the FMAs of
    the FP64 pipe.  These sums cancel, so they show what is rounded in single
    entries; the geometry's own rounding, the same for both, cancels in them."""
    path = os.path.join(str(tmp_path), "m.rom")
    romb.romb_train_gpu(0, 0, p, 4, n_r, 0.18, 0.44, LI.lhs(4 * n_r, 0.18, 0.44, seed=3), path)
    R = orom.read(path)
    lat = LI.lattice(12, 12, p, m, seed=5, mu_mode="graded", mu_range=(0.2, 0.42))
    nB, nd = (p + 1) ** 2, 2 * (p + 1) ** 2
    U = np.concatenate([np.asarray(R.I_pi)[:, None], np.asarray(R.U)], axis=1).reshape(nB, nB, 36, n_r + 1)
    T = U.reshape(nB, nB, 9, 2, 2, n_r + 1).transpose(1, 0, 2, 4, 3, 5).reshape(U.shape)
    lower = np.tri(nB, nB, -1, dtype=bool)[:, :, None, None]
    rows, diag = np.zeros((nB, 36, n_r + 1), np.longdouble), U[np.arange(nB), np.arange(nB)].astype(np.longdouble)
    for k in range(nB):   # sums over k2, of the half k1 <= k2 that the library holds
        rows += np.where(lower[:, k], T[:, k], U[:, k])
    C = [_chat(lat, c) for c in range(lat.ncells)]
    iu = np.triu_indices(nd)
    err = {}
    for pipe in (False, True):
        with romb.Context(0) as ctx:
            romb.romb_train_load(ctx.h, path)
            romb.romb_set_fp64_arithmetic(ctx.h, pipe)
            romb.romb_assemble(ctx.h, lat, romb.ROMB_FP64)
            K = romb.romb_read(ctx.h, "K").reshape(lat.ncells, -1)
            th = romb.romb_read(ctx.h, "theta").reshape(lat.ncells, -1)[:, :n_r + 1]
        e_row, e_net = [], []
        for c in range(lat.ncells):
            M = np.zeros((nd, nd), np.longdouble)
            M[iu] = K[c]
            M[(iu[1], iu[0])] = K[c]
            got = M.reshape(nB, 2, nB, 2).sum(axis=2)                                           # [k1][i1][i2]
            t = th[c].astype(np.longdouble)
            ref = np.einsum("akjl,kjlim->aim", (rows @ t).reshape(nB, 9, 2, 2), C[c])
            D = np.einsum("akjl,kjlim->aim", (diag @ t).reshape(nB, 9, 2, 2), C[c])
            ref[:, 1, 0] += D[:, 0, 1] - D[:, 1, 0]   # K holds its upper half
            e = ((got - ref) / np.abs(K[c]).max()).astype(float)
            e_row.append(np.mean(e ** 2))
            e_net.append(np.mean(e.sum(axis=0) ** 2))
        err[pipe] = np.sqrt([np.mean(e_row), np.mean(e_net)])
    assert np.all(err[False] <= err[True]), (err[False], err[True])
