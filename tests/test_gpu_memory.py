"""The integers of the FP64 kernels where memory is short: fields in pieces, no integers at all, and allocations that
fail in the middle of a call."""
import numpy as np
import pytest

from oracle import lattice as L
from paper_1903_06986_gb300 import lqcd, synth
from tests.gpu_util import context, dev, host, rel_err, torch_cuda

pytestmark = pytest.mark.gpu

KAPPA = 0.12
GIB = 1 << 30


def field(dims, n, seed):
    r = np.random.default_rng(seed)
    shp = L.field_shape(dims, (n,))
    return r.standard_normal(shp) + 1j * r.standard_normal(shp)


def links_bytes(V):
    return -(-V // 32) * 32 * 576 + 16 * V


def field_bytes(V):
    return -(-V // 32) * 32 * 192 + 4 * V


@pytest.mark.parametrize("fields", [1, 3, 0])
def test_pieces_of_a_block(fields):
    """Blocks converted one or three fields at a time give the bits of the whole block; without integers FP64."""
    torch = torch_cuda()
    dims, n = (4, 3, 5, 6), 7
    full, eo_dims = context(dims), (4, 6, 2, 4)
    U, Ue = dev(synth.su3_links(dims, 0.45, 1)), dev(synth.su3_links(eo_dims, 0.45, 2))
    x, eta, xe = dev(field(dims, n, 3)), dev(field(dims, n, 4)), dev(field(eo_dims, n, 5))
    eo = lqcd.EvenOddContext(eo_dims)
    e, o = eo.split(xe)

    def results():
        out = [full.wilson_apply(U, KAPPA, x, flags=f) for f in range(4)]
        out += [torch.from_numpy(full.contract(U, KAPPA, eta, x)), eo.hop(Ue, o, 0), eo.hop(Ue, e, 1), eo.rhs(Ue, KAPPA, xe),
                eo.reconstruct(Ue, KAPPA, e, xe)]
        return out + [eo.wilson_apply(Ue, KAPPA, e, flags=f) for f in range(4)]

    want = results()
    full.set_integer_workspace(fields * field_bytes(360), 0)
    eo.set_integer_workspace(fields * field_bytes(96), 0)
    assert full.workspace_bytes < links_bytes(360) + 4 * field_bytes(360) + (1 << 20)
    for i, (got, ref) in enumerate(zip(results(), want)):
        if fields:
            assert torch.equal(got, ref), i
        else:
            assert (got - ref).abs().max().item() <= 1e-13 * ref.abs().max().item(), i


def test_gives_everything_back():
    dims = (4, 4, 4, 4)
    ctx = context(dims)
    U, x = dev(synth.su3_links(dims, 0.45, 1)), dev(field(dims, 2, 3))
    ctx.gmresdr_solve(U, KAPPA, x, 20, 5, 1e-10, max_cycles=20)
    held = ctx.workspace_bytes
    ctx.set_integer_workspace(0, 0)
    assert ctx.workspace_bytes <= held - links_bytes(256) - 2 * field_bytes(256) - 21 * 2 * field_bytes(256)


@pytest.mark.parametrize("evenodd", [False, True])
@pytest.mark.parametrize("room", ["no links", "five fields", "fields, no basis"])
def test_solve_when_the_integers_do_not_fit(room, evenodd):
    """What fits is decided before a cycle is captured and kept for the call: the solve ends as it does with
    memory, and a later call with memory again takes the integers."""
    dims, n = (4, 4, 4, 6), 16
    full = context(dims)
    ctx = lqcd.EvenOddContext(dims) if evenodd else full
    U, b = synth.su3_links(dims, 0.45, 4), field(dims, n, 5)
    Ud = dev(U)
    bd = ctx.rhs(Ud, KAPPA, dev(b)) if evenodd else dev(b)
    V = 192 if evenodd else 384
    solve = lambda: ctx.gmresdr_solve(Ud, KAPPA, bd, 24, 6, 1e-12, max_cycles=40)
    want, info, _ = solve()                      # every workspace of the call
    ctx.set_integer_workspace(0, 0)
    plain, pinfo, _ = solve()
    held = ctx.workspace_bytes
    ctx.set_integer_workspace(GIB, GIB)
    more = {"no links": 1000, "five fields": links_bytes(384) + 5 * field_bytes(V) + 1000,
            "fields, no basis": links_bytes(384) + n * field_bytes(V) + 1000}[room]
    ctx.inject_memory_limit(held + more)
    got, ginfo, _ = solve()
    assert ginfo["converged"] and pinfo["converged"] and info["converged"]
    assert ctx.workspace_bytes <= held + more
    ctx.inject_memory_limit(0)
    again, _, _ = solve()
    assert torch_cuda().equal(again, want)
    for x in (plain, got):
        assert rel_err(host(x), host(want)) < 1e-10


def test_another_allocation_takes_the_room_of_the_integers():
    """Eigenvectors that fit only without the integer basis, then only without fields and links; what does not
    fit at all is refused, and the solve gives its bits again afterwards."""
    dims, k = (4, 4, 4, 6), 6
    ctx = context(dims)
    U, b = dev(synth.su3_links(dims, 0.45, 4)), dev(field(dims, 4, 5))
    E, lam = dev(field(dims, k, 6)), np.linspace(0.1, 0.6, k).astype(complex)
    solve = lambda: ctx.gmresdr_solve(U, KAPPA, b, 24, 6, 1e-12, max_cycles=40)[0]
    want, need = solve(), k * 12 * 384 * 16
    basis, fields = 25 * 4 * field_bytes(384), links_bytes(384) + 4 * field_bytes(384)
    assert need < fields < basis
    held = ctx.workspace_bytes
    ctx.inject_memory_limit(held + need - 1)
    d1 = ctx.defl_import(E, lam)
    assert ctx.workspace_bytes <= held - basis
    ctx.inject_memory_limit(ctx.workspace_bytes + need - 1)
    d2 = ctx.defl_import(E, lam)
    assert ctx.workspace_bytes <= held - basis - fields
    ctx.inject_memory_limit(ctx.workspace_bytes + need - 1)
    with pytest.raises(lqcd.LqcdError, match="status 6"):
        ctx.defl_import(E, lam)
    ctx.inject_memory_limit(0)
    assert torch_cuda().equal(solve(), want)
    d1.close(), d2.close()


def test_the_full_context_takes_the_room_of_its_reduced_one():
    """The integers that an even/odd loop's reduced context keeps make room for the full context."""
    dims, k = (4, 4, 4, 4), 6
    ctx = context(dims)
    U = dev(synth.su3_links(dims, 0.45, 2))
    E, lam = dev(field(dims, k, 6)), np.linspace(0.1, 0.6, k).astype(complex)
    loop = ctx.loop_setup(U, KAPPA, 3, 4, 4, 30, 8, 3, 3, 1e-10, 1e-10, evenodd=1)
    try:
        want = loop.noises(U, 0, 4)[0]
        ctx.set_integer_workspace(0, 0)              # of both
        bare = ctx.workspace_bytes
        ctx.set_integer_workspace(GIB, GIB)
        assert np.array_equal(loop.noises(U, 0, 4)[0], want)
        held, own = ctx.workspace_bytes, links_bytes(256) + 4 * field_bytes(256)
        assert held - bare > own + links_bytes(256) + field_bytes(128)      # both hold some
        ctx.inject_memory_limit(bare + k * 12 * 256 * 16 + 1000)
        ctx.defl_import(E, lam).close()
        assert ctx.workspace_bytes <= bare + 1000
        ctx.inject_memory_limit(0)
        assert np.array_equal(loop.noises(U, 0, 4)[0], want)
    finally:
        loop.close()
