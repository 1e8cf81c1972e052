"""Entries at the ends of the FP64 range, and far apart within a site, through the kernels that run on integers."""
import numpy as np
import pytest

from oracle import lattice as L, operators as O
from paper_1903_06986_gb300 import synth
from tests.gpu_util import context, dev, host, rel_err

pytestmark = pytest.mark.gpu


def field(dims, n, seed):
    r = np.random.default_rng(seed)
    shp = L.field_shape(dims, (n,))
    return r.standard_normal(shp) + 1j * r.standard_normal(shp)


@pytest.mark.parametrize("scale", [2.0 ** 970, 2.0 ** 1010, 2.0 ** -1000])
def test_contract_where_eta_times_the_integers_leaves_fp64(scale):
    """Finite densities although |eta| 2^62 is beyond the largest double (2^970, 2^1010), or eta is tiny."""
    dims = (3, 4, 2, 5)
    ctx = context(dims)
    U, eta, w = synth.su3_links(dims, 0.5, 1), field(dims, 2, 2), field(dims, 2, 3)
    eta[1] *= scale
    got = ctx.contract(dev(U), 0.14, dev(eta), dev(w))
    ref = O.per_t(O.densities(U, 0.14, eta / np.array([1.0, scale]).reshape(2, 1, 1, 1, 1, 1, 1), w)).transpose(1, 0, 2)
    assert np.isfinite(got).all()
    assert rel_err(got[0], ref[0]) < 1e-13
    assert rel_err(got[1] / scale, ref[1]) < 1e-13


KAPPA, EPS = 0.157, 2.0 ** -53


def abs_hop(U, psi):
    """sum over the directions of |1 -+ gamma| |U| |psi|: what roundings of the FP64 stencil are relative to."""
    a, out = np.abs(psi), 0.0
    for mu in range(4):
        m, p = np.abs(L.ONE4 - L.G[mu]), np.abs(L.ONE4 + L.G[mu])
        out = out + L.spin_apply(m, L.color_apply(np.abs(U[mu]), L.shift(a, mu, +1)))
        out = out + L.shift(L.spin_apply(p, L.color_apply_dag(np.abs(U[mu]).astype(complex), a)), mu, -1)
    return np.abs(out)


def around(dims, psi):
    """Largest real of the neighbours of each site, and the smallest such largest real that is not zero."""
    big = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(axis=(-1, -2))[..., None, None]
    nb = np.stack([L.shift(big, mu, s) for mu in range(4) for s in (+1, -1)])
    return nb.max(0), np.where(nb > 0, nb, np.inf).min(0)


def links(dims, kind):
    U = synth.su3_links(dims, 0.4323, 5)
    if kind != "su3":
        U = np.broadcast_to(np.eye(3, dtype=complex), U.shape).copy()
    if kind == "weak":
        r = np.random.default_rng(6)
        U += 1e-7 * (r.standard_normal(U.shape) + 1j * r.standard_normal(U.shape))
    return U


def spread(dims, n, kind):
    r = np.random.default_rng(7)
    psi = field(dims, n, 8)
    if kind == "within a site":        # 14 decades between the entries of a site
        psi *= 10.0 ** -r.uniform(0, 14, psi.shape)
    if kind == "reals":                # real and imaginary parts nine decades apart
        psi = psi.real + 1e-9j * psi.imag
    if kind == "spins":
        psi[..., 1, :] *= 1e-8
    if kind == "sites":                # neighbours 2^-20 of each other
        psi *= np.where(r.random(psi.shape[:5]) < 0.5, 1.0, 2.0 ** -20)[..., None, None]
    if kind == "point":
        psi[:] = 0.0
        psi[:, 1, 0, 1, 2, 2, 1] = 1.0 - 0.5j
    return psi


@pytest.mark.parametrize("kind", ["within a site", "reals", "spins", "sites", "point"])
@pytest.mark.parametrize("glue", ["unit", "weak", "su3"])
@pytest.mark.parametrize("dims,n", [((4, 3, 4, 5), 2), ((8, 8, 8, 16), 5)])
def test_operator_keeps_entries_far_below_the_largest(dims, n, glue, kind):
    """Entry by entry to FP64 roundings, in both launch forms (one thread per site, four warps per 32 sites), where
    entries, links or neighbours lie further apart than the integers hold them; closer ones to the
    integers' unit relative to 2^9 of the smallest neighbour (products at most 2^8 apart, one bit of the mantissas)."""
    ctx = context(dims)
    U, psi = links(dims, glue), spread(dims, n, kind)
    got = host(ctx.wilson_apply(dev(U), KAPPA, dev(psi)))
    ref = L.wilson(U.astype(np.clongdouble), np.longdouble(KAPPA), psi.astype(np.clongdouble))
    top, low = around(dims, psi)
    m = 0.0 if glue == "weak" or kind in ("within a site", "reals", "spins") else np.minimum(top, 2.0 ** 9 * low)
    m = np.where(np.isfinite(m), m, 0.0)
    # FP64: at most 24 + 8 + 2 roundings in a chain; integers: as in test_gpu_fxhop
    tol = 40 * EPS * (np.abs(psi) + KAPPA * abs_hop(U, psi)) + KAPPA * 8 * 6 * 2.0 ** -54 * m
    assert (np.abs(got - ref) <= tol).all()


@pytest.mark.parametrize("kind", ["within a site", "spins"])
def test_evenodd_hop_keeps_small_entries(kind):
    from paper_1903_06986_gb300 import lqcd
    dims = (4, 6, 4, 2)
    context(dims)
    ctx = lqcd.EvenOddContext(dims)
    U, psi = links(dims, "unit"), spread(dims, 3, kind)
    e, o = ctx.split(dev(psi))
    ref = host(ctx.split(dev(L.hop(U.astype(np.clongdouble), psi.astype(np.clongdouble)).astype(complex)))[0])
    tol = host(ctx.split(dev(abs_hop(U, psi).astype(complex)))[0]).real
    assert (np.abs(host(ctx.hop(dev(U), o, 0)) - ref) <= 41 * EPS * tol).all()


def test_contract_keeps_small_entries_of_w():
    """eta picks the small entries of w alone: point-split densities relative to them."""
    dims = (4, 3, 4, 6)
    ctx = context(dims)
    U, w = links(dims, "unit"), field(dims, 2, 9)
    w[..., :, 1] *= 1e-8                                   # one colour; unit links do not mix them
    eta = np.zeros_like(w)
    eta[..., :, 1] = field(dims, 2, 10)[..., :, 1]
    got = ctx.contract(dev(U), 0.14, dev(eta), dev(w))
    ref = O.per_t(O.densities(U, 0.14, eta, w)).transpose(1, 0, 2)
    assert rel_err(got, ref) < 1e-13


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("what", ["w", "eta", "links"])
def test_contract_with_a_non_finite_entry(what, bad):
    """The densities of the timeslices that the entry reaches are not finite, all others are those without it."""
    dims = (3, 4, 5, 6)
    ctx = context(dims)
    U, eta, w = synth.su3_links(dims, 0.5, 1), field(dims, 3, 2), field(dims, 3, 3)
    eta[2, 3], w[2, 0] = 0.0, 0.0                          # blocks of zeros beside it
    dens = lambda: O.per_t(O.densities(U, 0.14, eta, w)).transpose(1, 0, 2)
    at, clean = ((3, 2, 1, 0, 2, 1, 1) if what == "links" else (1, 2, 1, 0, 2, 3, 1)), dens()
    a = {"links": U, "eta": eta, "w": w}[what]
    a[at] += 1.0 - 2.0j
    fin = dens() == clean                                  # the projectors of t drop half of the spins
    a[at] = bad
    got = ctx.contract(dev(U), 0.14, dev(eta), dev(w))
    assert not fin.all() and np.array_equal(np.isfinite(got), fin)
    assert np.abs(got - clean)[fin].max() <= 1e-13 * np.abs(clean).max()


@pytest.mark.parametrize("kind", ["within a site", "sites", "point"])
def test_both_launch_forms_give_the_same_bits(kind):
    """Ten fields (a thread per site) and each of them alone (four warps per 32 sites), sites in FP64 among them."""
    from paper_1903_06986_gb300 import lqcd
    torch = pytest.importorskip("torch")
    dims, n = (8, 8, 8, 16), 10
    ctx, eo = context(dims), lqcd.EvenOddContext(dims)
    U, psi = dev(links(dims, "su3")), spread(dims, n, kind)
    psi[:, :5] = field(dims, n, 11)[:, :5]                 # timeslices of entries that the integers hold
    psi = dev(psi)
    for flag in range(4):
        whole = ctx.wilson_apply(U, KAPPA, psi, flags=flag)
        for r in (0, 7):
            assert torch.equal(ctx.wilson_apply(U, KAPPA, psi[r:r + 1].contiguous(), flags=flag)[0], whole[r]), (flag, r)
    e, o = eo.split(psi)
    for x, par in ((o, 0), (e, 1)):
        whole = eo.hop(U, x, par)
        assert torch.equal(eo.hop(U, x[3:4].contiguous(), par)[0], whole[3])


def few(dims, n, sites):
    """Gaussian fields with one entry 1e-9 of the others at the listed (t, z, y, x), and the mask of their neighbours."""
    psi, hit = field(dims, n, 12), np.zeros(field(dims, 1, 0).shape[1:5], bool)
    for i, at in enumerate(sites):
        psi[(slice(None),) + at + (i % 4, i % 3)] *= 1e-9
        hit[at] = True
    near = np.zeros_like(hit)
    for axis in range(4):
        near |= np.roll(hit, 1, axis) | np.roll(hit, -1, axis)
    return psi, near


FEW_SITES = [[(3, 2, 4, 5)], [(0, 0, 0, 0), (0, 0, 2, 1), (7, 1, 1, 1), (15, 7, 7, 7)],
             [(5, 5, y, x) for y in (0, 2, 4) for x in (0, 3, 6)]]


@pytest.mark.parametrize("n", [1, 6])
@pytest.mark.parametrize("sites", FEW_SITES)
def test_operator_with_few_sites_outside_the_integers(sites, n):
    """One, some and many lanes of a warp in FP64, entry by entry to its roundings; all forms of the operator."""
    from paper_1903_06986_gb300 import lqcd
    dims = (8, 8, 8, 16)
    ctx, eo = context(dims), lqcd.EvenOddContext(dims)
    U = links(dims, "su3")
    psi, near = few(dims, n, sites)
    g5 = lambda a: -a[..., [2, 3, 0, 1], :]
    ext = lambda a: L.wilson(U.astype(np.clongdouble), np.longdouble(KAPPA), a.astype(np.clongdouble))
    top, _ = around(dims, psi)
    m = np.where(near[..., None, None], 0.0, top)
    hopped, sum_abs = L.hop(U.astype(np.clongdouble), psi.astype(np.clongdouble)), abs_hop(U, psi)
    tol = 40 * EPS * (np.abs(psi) + KAPPA * sum_abs) + KAPPA * 8 * 6 * 2.0 ** -54 * m
    tol5 = 40 * EPS * (np.abs(g5(psi)) + KAPPA * abs_hop(U, g5(psi))) + KAPPA * 8 * 6 * 2.0 ** -54 * m
    for flag, ref, t in ((lqcd.APPLY_M, ext(psi), tol), (lqcd.APPLY_G5R, ext(g5(psi)), tol5),
                         (lqcd.APPLY_DAG, g5(ext(g5(psi))), np.abs(g5(tol5))),
                         (lqcd.APPLY_HOP, hopped, 40 * EPS * sum_abs + 8 * 6 * 2.0 ** -54 * m)):
        got = host(ctx.wilson_apply(dev(U), KAPPA, dev(psi), flags=flag))
        assert (np.abs(got - ref) <= t).all(), flag
    e, o = eo.split(dev(psi))
    want, bound = (eo.split(dev(a.astype(complex))) for a in (hopped, 41 * EPS * sum_abs + 8 * 6 * 2.0 ** -54 * m))
    for x, par in ((o, 0), (e, 1)):
        assert (np.abs(host(eo.hop(dev(U), x, par)) - host(want[par])) <= host(bound[par]).real).all(), par


@pytest.mark.parametrize("n", [1, 6])
@pytest.mark.parametrize("sites", FEW_SITES)
def test_contract_with_few_sites_outside_the_integers(sites, n):
    dims = (8, 8, 8, 16)
    ctx = context(dims)
    U, eta, (w, _) = links(dims, "su3"), field(dims, n, 13), few(dims, n, sites)
    got = ctx.contract(dev(U), 0.14, dev(eta), dev(w))
    ref = O.per_t(O.densities(U, 0.14, eta, w)).transpose(1, 0, 2)
    assert rel_err(got, ref) < 1e-13
