"""Gram-Schmidt on the integer form of the Krylov basis: solves whose vectors hold zeros, tiny and ragged
blocks of sites, several vector groups, restarts and block widths, against the dense solution or the
oracle's residual."""
import numpy as np
import pytest

from oracle import lattice as L
from paper_1903_06986_gb300 import lqcd, synth
from tests.gpu_util import context, dev, host, torch_cuda

pytestmark = pytest.mark.gpu

KAPPA = 0.12


def source(dims, n, kind, seed=21):
    r = np.random.default_rng(seed)
    shp = L.field_shape(dims, (n,))
    b = r.standard_normal(shp) + 1j * r.standard_normal(shp)
    if kind == "point":
        b[:] = 0.0
        for i in range(n):
            b[i, i % dims[3], 0, 1, 0, i % 4, i % 3] = 1.0
    if kind == "tiny sites":       # blocks that the integers do not hold: FP64 sums beside them
        b[:, 0] *= 1e-250
    if kind == "scales":
        b *= 10.0 ** r.integers(-12, 1, shp[:5])[..., None, None]
    return b


@pytest.mark.parametrize("kind", ["random", "point", "tiny sites", "scales"])
@pytest.mark.parametrize("dims,n,m,k", [((2, 2, 2, 4), 1, 24, 6), ((3, 5, 2, 7), 3, 13, 0), ((3, 5, 2, 7), 2, 20, 9)])
def test_gmresdr_solution(dims, n, m, k, kind):
    ctx = context(dims)
    U, b = synth.su3_links(dims, 0.45, 2), source(dims, n, kind)
    x, info, _ = ctx.gmresdr_solve(dev(U), KAPPA, dev(b), m, k, 3e-14, max_cycles=60)
    assert info["converged"]
    res = b - L.wilson(U, KAPPA, host(x))
    for i in range(n):
        assert np.linalg.norm(res[i]) <= 4e-14 * np.linalg.norm(b[i])


def test_arnoldi_relation_and_orthogonality():
    """The space that a solve returns: V orthonormal and A V_k = V_{k+1} Hbar to rounding, as with FP64 sums."""
    dims = (4, 4, 4, 6)
    ctx = context(dims)
    U = synth.su3_links(dims, 0.4323, 3)
    b = source(dims, 1, "random")
    for solve, op in ((ctx.gmresdr_solve, L.wilson), (ctx.minresdr_solve, L.wilson_g5)):
        _, _, d = solve(dev(U), KAPPA, dev(b), 40, 20, 1e-13, max_cycles=6, want_defl=True)
        e = d.export()
        V = host(e["V"])
        assert np.abs(V.conj() @ V.T - np.eye(len(V))).max() < 1e-13
        AV = op(U, KAPPA, V[:-1].reshape((-1,) + L.field_shape(dims, ()))).reshape(len(V) - 1, -1)
        assert np.abs(AV - e["Hbar"].T @ V).max() < 1e-13


def test_evenodd_block_and_mixed_operators():
    dims = (4, 6, 2, 4)
    context(dims)
    ctx = lqcd.EvenOddContext(dims)
    U, b = synth.su3_links(dims, 0.45, 4), source(dims, 9, "random")
    Ud = dev(U)
    be = ctx.rhs(Ud, KAPPA, dev(b))
    xe, info, _ = ctx.gmresdr_solve(Ud, KAPPA, be, 30, 8, 3e-14, max_cycles=40)
    assert info["converged"]
    x = host(ctx.reconstruct(Ud, KAPPA, xe, dev(b)))
    assert np.linalg.norm(b - L.wilson(U, KAPPA, x)) <= 1e-13 * np.linalg.norm(b)


def test_wide_ranges_of_block_widths_give_the_same_solutions():
    """50 right-hand sides of a block against the same ones alone: one and many chunks per inner product."""
    dims = (8, 8, 8, 8)
    torch = torch_cuda()
    ctx = context(dims)
    U, b = dev(synth.su3_links(dims, 0.4323, 5)), dev(source(dims, 17, "random"))
    x, info, _ = ctx.gmresdr_solve(U, KAPPA, b, 30, 10, 1e-13, max_cycles=40)
    assert info["converged"]
    for r in (0, 16):
        y, _, _ = ctx.gmresdr_solve(U, KAPPA, b[r:r + 1].contiguous(), 30, 10, 1e-13, max_cycles=40)
        assert (y[0] - x[r]).norm().item() <= 20 * 1e-13 * x[r].norm().item()
