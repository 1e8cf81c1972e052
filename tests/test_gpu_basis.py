"""The Gram-Schmidt kernels on the integer form of a basis (lqcd_basis_dot, lqcd_basis_update) against extended
precision: vector groups and their remainders, ragged blocks of sites, both forms of the update, sums at the
largest exponent growth, and entries that the integers do not hold."""
import numpy as np
import pytest

from oracle import lattice as L
from tests.gpu_util import context, dev, host

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def flat(a):
    return a.reshape(a.shape[:-6] + (-1, 12))          # (..., site, component)


def case(dims, nvec, nrhs, kind, seed=3):
    r = np.random.default_rng(seed)
    cplx = lambda shp: r.standard_normal(shp) + 1j * r.standard_normal(shp)
    V, w, h = cplx(L.field_shape(dims, (nvec, nrhs))), cplx(L.field_shape(dims, (nrhs,))), cplx((nvec, nrhs))
    if kind == "same sign":            # every term of a sum at the top of its exponent
        V[:], h[:], w[:] = 1.999 - 1.999j, 1.998, 1.999 + 1.999j
    if kind == "scales":               # sites, vectors and coefficients far apart, zero blocks, vectors and coefficients
        V *= 2.0 ** r.integers(-40, 40, V.shape[:6])[..., None, None]
        w *= 2.0 ** r.integers(-40, 40, w.shape[:5])[..., None, None]
        h *= 2.0 ** r.integers(-40, 40, h.shape)
        V[0, :, 0], h[-1] = 0.0, 0.0
        w[0, -1] = 0.0
    if kind == "outside":              # blocks, and coefficients, that the integers do not hold: FP64 sums
        V[0, :, 0] *= 1e-260
        V[-1, :, :, 1] *= 1e160
        w[:, :, :, 0] *= 1e-300
        w[:, 1] *= 1e100
        h[nvec // 2] *= 1e-200
    return V, w, h


def mags(V, w, h):
    """Per (vector, right-hand side, site): the largest real of V, of w and of h."""
    big = lambda a: np.maximum(np.abs(a.real), np.abs(a.imag)).astype(np.longdouble)
    return big(flat(V)).max(-1), big(flat(w)).max(-1), big(h)


@pytest.mark.parametrize("kind", ["random", "same sign", "scales", "outside"])
@pytest.mark.parametrize("dims,nvec,nrhs", [((3, 5, 2, 7), n, 1) for n in (1, 4, 5, 8, 9, 65, 240, 512)] +
                         [((3, 5, 2, 7), 9, 3), ((2, 2, 2, 2), 3, 2), ((8, 8, 8, 16), 9, 3), ((8, 8, 8, 16), 65, 3)])
def test_products_and_updates(dims, nvec, nrhs, kind):
    ctx = context(dims)
    V, w, h = case(dims, nvec, nrhs, kind)
    Vl, wl = flat(V), flat(w)
    ext = lambda a: a.astype(np.clongdouble)
    mV, mw, mh = mags(V, w, h)
    dot = host(ctx.basis_dot(dev(V), dev(w)))
    S = Vl.shape[-2]
    for i in range(nvec):
        ref = (ext(Vl[i]).conj() * ext(wl)).sum(axis=(-1, -2))
        # a site: 24 dropped low products of a quarter unit, 48 truncated inputs of a sixteenth and 4 roundings of half a
        # unit, unit 2^-54 of the product of the largest entries; FP64 sites: 24 roundings.  The sum over the
        # sites: at most S / 128 + 12 + 2 log2 roundings of partial sums
        tol = ((11 * 2.0 ** -54 + 24 * 2 * U * (S / 128.0 + 40)) * (mV[i] * mw)).sum(-1)
        assert (np.abs(dot[i] - ref) <= tol + 1e-320).all(), i
    got = host(ctx.basis_update(dev(V), dev(h), dev(w)))
    ref, T, M = ext(wl), np.zeros(wl.shape[:2], np.longdouble), np.zeros(wl.shape[:2], np.longdouble)
    for i in range(nvec):
        ref = ref - ext(Vl[i]) * h[i][:, None, None]
        T += mV[i] * mh[i][:, None]
        M = np.maximum(M, mV[i] * mh[i][:, None])
    # per vector: 2 low products of a quarter unit and 2 truncations of a 32nd; unit 2^-53 of the largest term, coarser
    # where the sum needs room; FP64 sites: 4 roundings per vector of partial sums up to |w| + 2 T
    tol = (0.75 * nvec + 2) * U * (M + T / 16) + 4 * U * (np.abs(wl).max(-1) + 2 * T)
    if kind == "outside":
        tol = tol + 4 * nvec * U * (np.abs(wl).max(-1) + 2 * T)
    assert (np.abs(flat(got) - ref).max(-1) <= 2 * tol + 1e-320).all()


def plain(V, w, h):
    with np.errstate(all="ignore"):
        d = np.stack([(flat(V)[i].conj() * flat(w)).sum(axis=(-1, -2)) for i in range(len(V))])
        u = flat(w).copy()
        for i in range(len(V)):
            u = u - flat(V)[i] * h[i][:, None, None]
    return d, u


@pytest.mark.parametrize("where", ["V", "w", "h", "V against zero", "w against zero", "V tiny, w inf", "zero coefficient"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_entries_are_not_lost(bad, where):
    """Every product and every updated site that FP64 sums make non-finite is non-finite here, and no other."""
    dims, nvec, nrhs = (3, 2, 4, 5), 5, 2
    ctx = context(dims)
    V, w, h = case(dims, nvec, nrhs, "random")
    at = (1, 3, 1, 0, 2)                                # right-hand side 1, one site
    if where == "V":
        V[(2,) + at + (1, 2)] = bad
    if where == "w":
        w[at + (1, 2)] = bad
    if where == "h":
        h[2, 1] = bad
    if where == "V against zero":
        V[(2,) + at + (1, 2)] = bad
        w[at] = 0.0
    if where == "w against zero":
        V[(2,) + at] = 0.0
        w[at + (1, 2)] = bad
    if where == "V tiny, w inf":
        V[(2,) + at] *= 2.0 ** -400
        w[at + (1, 2)] = bad
    if where == "zero coefficient":
        V[(2,) + at + (1, 2)] = bad
        h[2, 1] = 0.0
    d, u = plain(V, w, h)
    with np.errstate(all="ignore"):
        assert np.array_equal(np.isfinite(host(ctx.basis_dot(dev(V), dev(w)))), np.isfinite(d))
        assert np.array_equal(np.isfinite(flat(host(ctx.basis_update(dev(V), dev(h), dev(w))))).all(-1),
                              np.isfinite(u).all(-1))


def test_denormal_blocks():
    """Sites whose entries are all below 2^-1022 (high word zero too) count as numbers, not as zeros."""
    dims, nvec = (2, 2, 2, 2), 2
    ctx = context(dims)
    V, w, h = case(dims, nvec, 1, "random")
    V[0, 0, 1] = 3e-320 + 1e-318j
    w[0, 1] *= 1e300
    V[1, 0, 0] *= 1e300
    w[0, 0] = 5e-321
    d, u = plain(V, w, h)
    got = host(ctx.basis_dot(dev(V), dev(w)))
    # the denormal site's share is far below the rounding of the others: alone, it is what is left
    V[0] = np.where(V[0] == V[0, 0, 1, 0, 0, 0, 0, 0], V[0], 0.0)
    want = plain(V, w, h)[0][0]
    alone = host(ctx.basis_dot(dev(V), dev(w)))[0]
    assert np.abs(got - d).max() <= 1e-13 * np.abs(d).max()
    assert np.abs(want).min() > 0 and np.abs(alone - want).max() <= 1e-12 * np.abs(want).max()


def test_arguments():
    from paper_1903_06986_gb300 import lqcd
    assert lqcd.load().lqcd_basis_dot(None, None, 1, None, 1, None) == lqcd.ERR_INVALID_ARG
    assert lqcd.load().lqcd_basis_update(None, None, 1, None, None, 1) == lqcd.ERR_INVALID_ARG


def test_a_tiny_site_with_zeros_against_a_large_one():
    """The zeros of a site whose largest entry is near 1e-300 stay zeros in products with entries of 2^200."""
    dims = (3, 2, 4, 5)
    ctx = context(dims)
    V, w, h = case(dims, 3, 1, "random")
    at = (0, 3, 1, 0, 2)
    V[(1,) + at] *= 2.0 ** 200
    w[:] = 0.0
    w[at + (2, 1)] = 1e-300 - 2e-300j
    d, _ = plain(V, w, h)
    assert np.abs(host(ctx.basis_dot(dev(V), dev(w))) - d).max() <= 1e-14 * np.abs(d).max()


@pytest.mark.parametrize("nvec", [1, 2, 7, 8, 11])
@pytest.mark.parametrize("prec,v,wv", [("f32", 1 + 2.0 ** -9, 1 + 2.0 ** -11), ("f16", 1 + 2.0 ** -10, 1 + 2.0 ** -10)])
def test_packed_products_of_equal_terms(prec, v, wv, nvec):
    """Terms 1 + 2^-9 + .. + 2^-20 of equal sign: a chain of FP32 additions drops the last part of each beyond 2^4
    (2^-21 of the sum and more); sums of at most 8 terms are exact, and their sum is off by a rounding per thread."""
    from paper_1903_06986_gb300 import lqcd
    dims, nrhs = (8, 8, 8, 16), 2
    ctx = context(dims)
    pr = {"f32": lqcd.PREC_F32, "f16": lqcd.PREC_F16}[prec]
    pack = (lambda x: ctx.pack_f32(x)) if prec == "f32" else (lambda x: ctx.pack_half(x, pr))
    V = dev(np.full(L.field_shape(dims, (nvec * nrhs,)), v * (1 + 1j)))
    w = dev(np.full(L.field_shape(dims, (nrhs,)), wv * (1 + 1j)))
    h = host(ctx.basis_dot_packed(pack(V), pack(w), nvec, nrhs, pr))
    want = 2 * v * wv * 12 * 8192
    assert np.abs(h - want).max() <= 2.0 ** -23 * want


@pytest.mark.parametrize("dims,nvec,nrhs", [((2, 2, 2, 2), 2, 1), ((4, 4, 4, 8), 8, 1), ((5, 3, 7, 9), 1, 2), ((5, 3, 7, 9), 9, 3),
                                            ((8, 8, 8, 16), 2, 1), ((12, 12, 12, 24), 2, 1), ((6, 6, 6, 12), 40, 12)])
@pytest.mark.parametrize("prec", ["f32", "f16"])
def test_packed_products_of_short_fields(prec, dims, nvec, nrhs):
    """Chunks of 8 elements per thread where 8 loads would leave SMs without a block, and their remainders."""
    from paper_1903_06986_gb300 import lqcd
    ctx = context(dims)
    pr = {"f32": lqcd.PREC_F32, "f16": lqcd.PREC_F16}[prec]
    pack = ctx.pack_f32 if prec == "f32" else lambda x: ctx.pack_half(x, pr)
    unpack = ctx.unpack_f32 if prec == "f32" else lambda x: ctx.unpack_half(x, pr)
    r = np.random.default_rng(21)
    make = lambda n: dev(r.standard_normal(L.field_shape(dims, (n,))) + 1j * r.standard_normal(L.field_shape(dims, (n,))))
    V, w = pack(make(nvec * nrhs)), pack(make(nrhs))
    got = host(ctx.basis_dot_packed(V, w, nvec, nrhs, pr))
    v, u = host(unpack(V)).reshape(nvec, nrhs, -1), host(unpack(w)).reshape(nrhs, -1)
    # FP32 chains of at most 8 products, a rounding of their sums, and those of the stored scale
    tol = 16 * 2.0 ** -24 * (np.abs(v) * np.abs(u)).sum(-1) * 2 ** 0.5
    assert (np.abs(got - (v.conj() * u).sum(-1)) <= tol).all()
