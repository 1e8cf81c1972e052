"""The fixed-point form of the FP64 Wilson operator against the oracle in extended precision, at the
sizes and values where it can go wrong: single warps and ragged tails, both launch forms, fields with
zeros, wide dynamic ranges and non-finite entries, odd directions of even/odd contexts, capture."""
import numpy as np
import pytest

from oracle import lattice as L
from paper_1903_06986_gb300 import synth
from tests.gpu_util import context, dev, host, torch_cuda

pytestmark = pytest.mark.gpu

FORMS = {0: L.wilson, 1: L.wilson_g5, 2: L.wilson_dag}
KAPPA = 0.157
EPS = 2.0 ** -53


def reference(U, psi, flag):
    Ul, pl = U.astype(np.clongdouble), psi.astype(np.clongdouble)
    return L.hop(Ul, pl) if flag == 3 else FORMS[flag](Ul, np.longdouble(KAPPA), pl)


def bound(psi, ref, flag):
    """Roundings of one output real: the sum's conversion to FP64, the last multiply-add and the result
    (three of them, 2^-53 of |hop| and |out| each), and per direction the dropped low product and the
    floor of the shift (2^-55 of the largest link real times the largest half-spinor real, at most
    2 times the largest real around; 6 products, 8 directions)."""
    big = np.abs(psi).max()
    k = 1.0 if flag == 3 else KAPPA
    return 3 * EPS * (np.abs(ref) + np.abs(psi if flag != 3 else 0) + k * 8) + k * 8 * 6 * 2.0 ** -54 * big


def field(dims, n, seed):
    r = np.random.default_rng(seed)
    shp = L.field_shape(dims, (n,))
    return r.standard_normal(shp) + 1j * r.standard_normal(shp)


@pytest.mark.parametrize("dims,n", [((2, 2, 2, 2), 1), ((3, 5, 2, 7), 2), ((4, 4, 4, 6), 3), ((6, 4, 5, 3), 12)])
@pytest.mark.parametrize("flag", [0, 1, 2, 3])
def test_error_against_extended_precision(dims, n, flag):
    ctx = context(dims)
    U, psi = synth.su3_links(dims, 0.4323, 5), field(dims, n, 6)
    got = host(ctx.wilson_apply(dev(U), KAPPA, dev(psi), flags=flag))
    ref = reference(U, psi, flag)
    err = (got - ref).astype(np.complex128)
    assert (np.abs(err) <= bound(psi, ref, flag)).all()
    # and in the 2-norm no further off than the FP64 stencil of the oracle
    plain = L.hop(U, psi) if flag == 3 else FORMS[flag](U, KAPPA, psi)
    assert np.linalg.norm(err) <= np.linalg.norm((plain - ref).astype(np.complex128))


def test_forms_and_blocks_agree_bit_for_bit():
    """One right-hand side at a time (four warps per 32 sites) and all together (one thread per site)."""
    dims, n = (8, 8, 8, 16), 12
    ctx = context(dims)
    Ud, p = dev(synth.su3_links(dims, 0.4323, 7)), dev(field(dims, n, 8))
    for flag in (1, 3):
        whole = ctx.wilson_apply(Ud, KAPPA, p, flags=flag)
        for r in (0, 5, n - 1):
            assert torch_cuda().equal(ctx.wilson_apply(Ud, KAPPA, p[r:r + 1].contiguous(), flags=flag)[0], whole[r])


def test_general_links_zeros_and_dynamic_range():
    dims = (4, 3, 2, 5)
    ctx = context(dims)
    r = np.random.default_rng(9)
    shp = synth.unit_links(dims).shape
    U = (r.standard_normal(shp) + 1j * r.standard_normal(shp)) * 3.0     # not unitary
    U[1, 2] = 0.0
    psi = field(dims, 3, 10)
    psi[1] *= 2.0 ** r.integers(-300, 300, psi[1].shape[:4])[..., None, None]   # sites far apart in scale
    psi[2] = 0.0
    psi[2, 1, 0, 2, 3, 2, 1] = 1.0
    got = host(ctx.wilson_apply(dev(U), KAPPA, dev(psi), flags=0))
    ref = reference(U, psi, 0).astype(np.complex128)
    # per output site: relative to the largest entry around it (itself and its neighbours)
    mag = np.abs(psi).max(axis=(-2, -1)) * np.abs(U).max() * 8 + 1e-300
    around = mag.copy()
    for ax in range(1, 5):
        around = np.maximum.reduce([around, np.roll(mag, 1, ax), np.roll(mag, -1, ax)])
    assert (np.abs(got - ref).max(axis=(-2, -1)) <= 64 * EPS * around).all()
    assert not got[2][np.abs(ref[2]) == 0].any()


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e300, 1e-300, 5e-324])
def test_entries_outside_the_fixed_point_range(bad):
    """NaN, Inf and extreme magnitudes give what the FP64 stencil gives, and nothing leaks to sites more
    than one hop away."""
    dims = (4, 4, 4, 4)
    ctx = context(dims)
    U, psi = synth.su3_links(dims, 0.4323, 11), field(dims, 1, 12)
    psi[0, 1, 2, 3, 0] = bad
    clean = psi.copy()
    clean[0, 1, 2, 3, 0] = 0.0
    got, base = (host(ctx.wilson_apply(dev(U), KAPPA, dev(f)))[0] for f in (psi, clean))
    with np.errstate(all="ignore"):
        ref = L.wilson(U, KAPPA, psi)[0]
    d = np.zeros(L.site_shape(dims), dtype=int)
    for ax, at in enumerate((1, 2, 3, 0)):
        c = np.abs(np.arange(4) - at)
        d = d + np.minimum(c, 4 - c).reshape([-1 if a == ax else 1 for a in range(4)])
    assert np.array_equal(got[d > 1], base[d > 1])
    near = got[d <= 1]
    if np.isfinite(bad):
        scale = max(abs(bad), 1.0)
        assert np.abs(near - ref[d <= 1]).max() <= 64 * EPS * 8 * scale
    else:
        assert not np.isfinite(near).all()
    U2 = U.copy()
    U2[2, 0, 1, 1, 1] = np.nan
    assert np.isnan(host(ctx.wilson_apply(dev(U2), KAPPA, dev(clean)))[0, 0, 1, 1, 1]).any()


def test_under_capture_and_on_another_stream():
    """A caller's graph capture takes the stencil without workspace; a context moved to another stream
    waits for its converted links."""
    torch = torch_cuda()
    dims = (4, 4, 4, 8)
    ctx = context(dims)
    Ud, p = dev(synth.su3_links(dims, 0.4323, 13)), dev(field(dims, 2, 14))
    want, out = ctx.wilson_apply(Ud, KAPPA, p), torch.empty_like(p)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    fresh = context(dims)
    with torch.cuda.graph(g, stream=side):
        fresh.set_stream(torch.cuda.current_stream().cuda_stream)
        fresh.wilson_apply(Ud, KAPPA, p, out=out)
    g.replay()
    torch.cuda.synchronize()
    assert (out - want).abs().max().item() <= 16 * EPS * 8
    for s in (side, torch.cuda.Stream(), side):
        ctx.set_stream(s.cuda_stream)
        out.zero_()
        s.wait_stream(torch.cuda.current_stream())
        ctx.wilson_apply(Ud, KAPPA, p, out=out)
        torch.cuda.synchronize()
        assert torch.equal(out, want)


@pytest.mark.parametrize("dims", [(2, 4, 2, 6), (6, 4, 4, 2)])
def test_evenodd_forms(dims):
    from paper_1903_06986_gb300 import lqcd
    context(dims)
    ctx = lqcd.EvenOddContext(dims)
    U, psi = synth.su3_links(dims, 0.4323, 15), field(dims, 2, 16)
    Ud, pd = dev(U), dev(psi)
    e, o = ctx.split(pd)
    hop = reference(U, psi, 3)
    for par, inp in ((0, o), (1, e)):
        got = host(ctx.hop(Ud, inp, par))
        z = torch_cuda().zeros_like(e)
        other = host(ctx.split(dev(hop.astype(np.complex128)))[par])
        assert np.abs(got - other).max() <= 6 * EPS * 16 + 8 * 6 * 2.0 ** -54 * np.abs(psi).max(), par
        assert not host(ctx.hop(Ud, z, par)).any()
