"""Launch forms that depend on sizes, where they can go wrong: right-hand sides split over a block in the
link gradient, chunks of a timeslice in the contraction, hopping traces by site."""
import numpy as np
import pytest

from oracle import derivs as Dv, lattice as L, operators as O, subtract as S
from paper_1903_06986_gb300 import lqcd, synth
from tests.gpu_util import context, dev, host, rel_err

pytestmark = pytest.mark.gpu


def fields(dims, n, seed):
    r = np.random.default_rng(seed)
    shp = L.field_shape(dims, (n,))
    return r.standard_normal(shp) + 1j * r.standard_normal(shp)


@pytest.mark.parametrize("dims,n", [((3, 2, 4, 4), 1), ((3, 2, 4, 4), 4), ((2, 3, 5, 2), 7), ((4, 4, 4, 3), 5)])
def test_link_grad_groups(dims, n):
    """n = 1: one thread per link; else four groups of right-hand sides, the last ones short."""
    ctx = context(dims)
    U, x, z = synth.su3_links(dims, 0.5, 3), fields(dims, n, 1), fields(dims, n, 2)
    g, gl = lqcd.link_grad(ctx, dev(U), 0.137, dev(z), dev(x), scale=0.5)
    ref = 0.5 * sum(Dv.link_gradient(U, 0.137, x[r], z[r]) for r in range(n))
    assert rel_err(host(g), ref) < 1e-12
    dU = sum(Dv.link_matrix_derivatives(U, 0.137, x[r], z[r])[0] for r in range(n))
    dUc = sum(Dv.link_matrix_derivatives(U, 0.137, x[r], z[r])[1] for r in range(n))
    assert rel_err(host(gl), 0.5 * (dUc + dU.conj())) < 1e-12


def test_link_grad_one_call_is_the_sum_of_single_ones():
    """20736 sites: one thread per link with every right-hand side in it, against n calls of one."""
    dims, n = (12, 12, 12, 12), 5
    ctx = context(dims)
    Ud, x, z = dev(synth.su3_links(dims, 0.4323, 4)), dev(fields(dims, n, 5)), dev(fields(dims, n, 6))
    g, gl = lqcd.link_grad(ctx, Ud, 0.137, z, x)
    parts = [lqcd.link_grad(ctx, Ud, 0.137, z[r:r + 1].contiguous(), x[r:r + 1].contiguous()) for r in range(n)]
    for got, i in ((g, 0), (gl, 1)):
        want = sum(host(p[i]) for p in parts)
        assert rel_err(host(got), want) < 1e-14


@pytest.mark.parametrize("dims,n", [((9, 7, 11, 3), 2), ((16, 16, 8, 2), 1), ((5, 3, 2, 6), 40)])
def test_contract_chunks(dims, n):
    """Ragged chunks of a timeslice (the last one short), several chunks with few pairs, one with many."""
    ctx = context(dims)
    U, eta, w = synth.su3_links(dims, 0.5, 7), fields(dims, n, 8), fields(dims, n, 9)
    got = ctx.contract(dev(U), 0.14, dev(eta), dev(w))
    ref = O.per_t(O.densities(U, 0.14, eta, w)).transpose(1, 0, 2)
    assert rel_err(got, ref) < 1e-13


@pytest.mark.parametrize("dims,K", [((3, 3, 3, 3), 2), ((4, 5, 4, 6), 3), ((5, 5, 6, 5), 4), ((6, 8, 6, 7), 5),
                                    ((7, 7, 7, 8), 6), ((8, 8, 8, 9), 7), ((9, 9, 9, 10), 8)])
def test_hop_traces_by_site(dims, K):
    """Extents just above K (no walk of the trace winds) and odd ones: source by source against the
    probing form with every order a full application, order by order."""
    ctx = context(dims)
    Ud = dev(synth.su3_links(dims, 0.5, 11))
    got = ctx.hop_traces(Ud, 0.13, K)
    ctx.set_probe_depth(max(1, K - 1))
    want = ctx.hop_traces(Ud, 0.13, K)
    # order k sums V terms of size up to 8^k / ... : relative to the largest entry of the order, or to the
    # rounding of the 12 V unit terms where the order vanishes
    for k in range(K):
        scale = max(np.abs(want[k]).max(), 12.0 * np.prod(dims[:3]) * 2.0 ** k)
        assert np.abs(got[k] - want[k]).max() <= 1e-13 * scale, k


def test_hop_traces_by_site_against_the_oracle():
    dims, K = (4, 4, 4, 4), 3
    ctx = context(dims)
    U = synth.su3_links(dims, 0.5, 12)
    assert rel_err(ctx.hop_traces(dev(U), 0.13, K), O.per_t(S.hop_traces(U, 0.13, K, dims))) < 1e-13


@pytest.mark.parametrize("prec,eps", [(lqcd.PREC_F16, 2.0 ** -11), (lqcd.PREC_BF16, 2.0 ** -8)])
def test_packed_register_forms(prec, eps):
    """Six fields of 12^3 x 24 are more than two waves of the wide form's blocks, a pair of them less: each pair
    against the same fields in the block, to one rounding of the storage."""
    dims, n = (12, 12, 12, 24), 6
    ctx = context(dims)
    Up = ctx.pack_links_f32(dev(synth.su3_links(dims, 0.4323, 13)), 12)
    p = ctx.pack_half(dev(fields(dims, n, 14)), prec)
    for flag in (0, 1, 2, 3):
        whole = host(ctx.unpack_half(ctx.wilson_apply_half(Up, 12, 0.137, p, flags=flag, prec=prec), prec))
        for r in (0, 4):
            pair = host(ctx.unpack_half(ctx.wilson_apply_half(Up, 12, 0.137, p[r:r + 2].contiguous(), flags=flag,
                                                              prec=prec), prec))
            for a, b in ((pair.real, whole[r:r + 2].real), (pair.imag, whole[r:r + 2].imag)):
                assert (np.abs(a - b) <= 2 * eps * np.abs(b) + 1e-7 * np.abs(whole).max()).all()


def test_hop_traces_by_site_at_its_last_order():
    """K = 9, the largest that is followed source by source: gauge-rotated unit links, whose traces are those of the
    free field, and general links against the probing form."""
    from tests.test_oracle_traces import free_hop_traces
    dims, K = (10, 10, 11, 10), 9
    ctx = context(dims)
    r = np.random.default_rng(15)
    g = np.linalg.qr(r.standard_normal((10, 11, 10, 10, 3, 3)) + 1j * r.standard_normal((10, 11, 10, 10, 3, 3)))[0]
    U = np.stack([g @ np.roll(g, -1, axis=3 - mu).conj().swapaxes(-1, -2) for mu in range(4)])
    got, ref = ctx.hop_traces(dev(U), 0.13, K).sum(axis=-1), free_hop_traces(dims, 0.13, K)
    ref[np.abs(ref) < 1e-3] = 0.0   # zeros of the momentum sum to its rounding; the others are at least 12 V kappa
    scale = 12.0 * np.prod(dims) * 2.0 ** np.arange(K)
    assert (np.abs(got - ref).max(axis=-1) <= 1e-13 * np.maximum(np.abs(ref).max(axis=-1), scale)).all()
    Ud = dev(synth.su3_links(dims, 0.5, 16))
    got = ctx.hop_traces(Ud, 0.13, K)
    ctx.set_probe_depth(K - 1)
    want = ctx.hop_traces(Ud, 0.13, K)
    for k in range(K):
        scale = max(np.abs(want[k]).max(), 12.0 * np.prod(dims[:3]) * 2.0 ** k)
        assert np.abs(got[k] - want[k]).max() <= 1e-13 * scale, k


@pytest.mark.parametrize("recon", [12, 18])
def test_packed_block_sizes(recon):
    """FP32 fields of 12^3 x 24 in blocks of 128 threads (four fields, a wave), of 64 (two; ten) and of a ragged lattice:
    the same bits in every block."""
    torch = pytest.importorskip("torch")
    for dims, sizes in (((12, 12, 12, 24), (10, 4, 2)), ((13, 11, 15, 17), (5, 2))):
        ctx = context(dims)
        Up = ctx.pack_links_f32(dev(synth.su3_links(dims, 0.4323, 13)), recon)
        p = ctx.pack_f32(dev(fields(dims, sizes[0], 14)))
        for flag in range(4):
            whole = ctx.wilson_apply_packed(Up, recon, 0.137, p, flags=flag)
            for n in sizes[1:]:
                part = ctx.wilson_apply_packed(Up, recon, 0.137, p[:n].contiguous(), flags=flag)
                assert torch.equal(part, whole[:n]), (dims, n, flag)
