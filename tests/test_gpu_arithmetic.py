"""romb_set_fp64_arithmetic: what it reaches, and that it stays the caller's."""
import numpy as np
import pytest

import lattice_inputs as LI

from romb_testutil import small_rom, unpack_upper

pytestmark = pytest.mark.gpu
romb = pytest.importorskip("paper_2604_09113_gb300")
torch = pytest.importorskip("torch")
from paper_2604_09113_gb300.autograd import compliance  # noqa: E402

U = 2.0 ** -53


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


@pytest.mark.parametrize("precision", ["ROMB_FP64", "ROMB_FP32_SPLIT"])
def test_without_a_choice_a_gradient_holds_for_its_lattice(precision):
    """Where nobody chose, a gradient in the FP64 form takes the FP64 pipe for the
    lattices of its shape; another shape, and a split form, leave the default.  A
    choice made afterwards holds."""
    lat, other = _lat(4), _lat(4, 3, 3)
    _, path = small_rom(0, 4, 0.18, 0.40, 20, 12, 1)
    with romb.Context(0) as ctx:
        romb.romb_train_load(ctx.h, path)
        default, default_other = _k(ctx, lat), _k(ctx, other)
        ctrl = torch.tensor(lat.ctrl, requires_grad=True)
        mu = torch.tensor(lat.mu, requires_grad=True)
        compliance(ctx, lat, ctrl, mu, getattr(romb, precision), rtol=1e-8).backward()
        assert np.array_equal(_k(ctx, lat), default) == (precision != "ROMB_FP64")
        assert np.array_equal(_k(ctx, other), default_other)
        bad = _lat(4, 3, 3)
        bad.rho = -1.0
        with pytest.raises(romb.RombError):   # a refused gradient leaves nothing behind
            compliance(ctx, bad, torch.tensor(bad.ctrl), torch.tensor(bad.mu), getattr(romb, precision), rtol=1e-8)
        assert np.array_equal(_k(ctx, lat), default)
        compliance(ctx, lat, ctrl, mu, getattr(romb, precision), rtol=1e-8).backward()
        romb.romb_set_fp64_arithmetic(ctx.h, False)
        assert np.array_equal(_k(ctx, lat), default)


@pytest.mark.parametrize("source", ["given", "ROMB_FP32_SPLIT", "ROMB_BF16_SPLIT"])
def test_choice_reaches_every_factorisation(source):
    """The factorisation of the caller's own matrices and of the split forms
    follows the choice, too: with the FP64 pipe S of the caller's matrices is,
    bit by bit, that of the same matrices assembled in the FP64 form."""
    p = 4
    lat = _lat(p)
    nd = 2 * (p + 1) ** 2
    _, path = small_rom(0, p, 0.18, 0.40, 20, 12, 1)
    S = {}
    with romb.Context(0) as ctx:
        romb.romb_train_load(ctx.h, path)
        romb.romb_set_fp64_arithmetic(ctx.h, True)
        K = np.stack([unpack_upper(k, nd) for k in _k(ctx, lat).reshape(lat.ncells, -1)])
        romb.romb_factor(ctx.h)
        own = romb.romb_read(ctx.h, "S")
        for pipe in (False, True):
            romb.romb_set_fp64_arithmetic(ctx.h, pipe)
            if source == "given":
                romb.romb_assemble_host_K(ctx.h, lat, K)
            else:
                romb.romb_assemble(ctx.h, lat, getattr(romb, source))
            romb.romb_factor(ctx.h)
            S[pipe] = romb.romb_read(ctx.h, "S")
    assert not np.array_equal(S[False], S[True])
    assert np.abs(S[False] - S[True]).max() <= 3 * 2 * (p - 1) ** 2 * U * np.abs(K).max()
    if source == "given":
        assert np.array_equal(S[True], own)


@pytest.mark.parametrize("p,n", [(3, 16), (4, 12), (5, 10), (6, 8), (7, 7), (8, 6)])
def test_both_arithmetics_at_every_degree(p, n):
    """K of both arithmetics agrees to rounding.  Of the same K, S of the default is
    no further (rms) from extended precision than that of the FP64 pipe, and the
    solves agree in iterations and displacement."""
    lat = _lat(p, n, n)
    nB, nd, nU = (p + 1) ** 2, 2 * (p + 1) ** 2, 8 * p
    _, path = small_rom(0, p, 0.18, 0.40, 20, 12, 1)
    k = np.arange(nB)
    bd = (k % (p + 1) == 0) | (k % (p + 1) == p) | (k < p + 1) | (k >= nB - p - 1)
    iU, iI = np.repeat(bd, 2).nonzero()[0], np.repeat(~bd, 2).nonzero()[0]
    nodes = (p * lat.nx + 1) * (p * lat.ny + 1)
    S, u, its = {}, {}, {}
    with romb.Context(0) as ctx:
        romb.romb_train_load(ctx.h, path)
        romb.romb_set_fp64_arithmetic(ctx.h, True)
        Kp = _k(ctx, lat).reshape(lat.ncells, -1)
        romb.romb_set_fp64_arithmetic(ctx.h, False)
        Kd = _k(ctx, lat).reshape(lat.ncells, -1)
        assert np.abs(Kd - Kp).max() <= 2 * 53 * U * np.abs(Kp).max()   # n_r + 41 roundings each
        romb.romb_factor(ctx.h)   # indefinite cells take the exact matrices
        K = np.stack([unpack_upper(v, nd) for v in romb.romb_read(ctx.h, "K").reshape(lat.ncells, -1)])
        for pipe in (False, True):
            romb.romb_set_fp64_arithmetic(ctx.h, pipe)
            romb.romb_assemble_host_K(ctx.h, lat, K)
            romb.romb_factor(ctx.h)
            S[pipe] = romb.romb_read(ctx.h, "S").reshape(lat.ncells, -1)
            u[pipe], its[pipe], _ = romb.romb_bddc_solve(ctx.h, nodes, rtol=1e-10, maxit=500)
    e2 = {False: 0.0, True: 0.0}
    for c in range(lat.ncells):
        if c % n == 0:
            continue   # clamped nodes
        A, W = K[c][np.ix_(iI, iI)].astype(np.longdouble), K[c][np.ix_(iI, iU)].astype(np.longdouble)
        for j in range(len(iI)):   # elimination of the interior
            f = A[j + 1:, j] / A[j, j]
            W[j + 1:] -= np.outer(f, W[j])
            A[j + 1:, j:] -= np.outer(f, A[j, j:])
        W /= np.sqrt(np.diag(A))[:, None]
        ref = K[c][np.ix_(iU, iU)] - W.T @ W
        d = np.sqrt(np.diag(K[c])[iU])
        for pipe in S:
            e2[pipe] += np.mean(((unpack_upper(S[pipe][c], nU) - ref).astype(float) / np.outer(d, d)) ** 2)
    assert e2[False] <= e2[True], e2
    assert list(its[False]) == list(its[True])
    assert np.abs(u[False] - u[True]).max() <= 1e-8 * np.abs(u[True]).max()
