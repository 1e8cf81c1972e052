"""Calls queued back to back on several streams of one context: the converted links and fields that they share are
not overwritten while an earlier call reads them."""
import ctypes

import numpy as np
import pytest

from oracle import lattice as L
from paper_1903_06986_gb300 import lqcd, synth
from tests.gpu_util import context, dev, torch_cuda

pytestmark = pytest.mark.gpu

KAPPA = 0.14


def field(dims, n, seed):
    r = np.random.default_rng(seed)
    shp = L.field_shape(dims, (n,))
    return dev(r.standard_normal(shp) + 1j * r.standard_normal(shp))


@pytest.mark.parametrize("kind", ["operator", "contract", "evenodd"])
def test_calls_on_alternating_streams(kind):
    """Blocks converted one field at a time (32 launches of some 20 us a call), different links and fields, no
    synchronisation between the calls: bit for bit the results of one call at a time."""
    torch = torch_cuda()
    dims, n = (12, 12, 12, 12), 16
    full = context(dims)
    ctx = lqcd.EvenOddContext(dims) if kind == "evenodd" else full
    ctx.set_integer_workspace(1, 0)
    Us = [dev(synth.su3_links(dims, 0.45, 20 + i)) for i in range(3)]
    xs = [field(dims, n, 30 + i) for i in range(3)]
    if kind == "evenodd":
        xs = [ctx.split(x)[1] for x in xs]
    outs = [torch.empty_like(x) for x in xs]

    def call(i):
        if kind == "evenodd":
            return ctx.hop(Us[i], xs[i], 0)
        return ctx.wilson_apply(Us[i], KAPPA, xs[i], out=outs[i])

    want = [call(i).clone() for i in range(3)]
    if kind == "contract":
        dens = full.contract(Us[1], KAPPA, xs[0], xs[1])
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(3)]
    got = []
    for rep in range(3):
        for i, s in enumerate(streams):
            ctx.set_stream(s.cuda_stream)
            if kind == "contract" and i == 1:       # between two operators; returns host data
                assert np.array_equal(full.contract(Us[1], KAPPA, xs[0], xs[1]), dens)
                continue
            got.append((i, call(i)))
    torch.cuda.synchronize()
    for i, g in got:
        assert torch.equal(g, want[i]), i


def test_a_new_stream_on_the_handle_of_a_destroyed_one():
    """cudaStreamDestroy returns before the stream's work ends, and the next stream may get its handle."""
    torch = torch_cuda()
    try:
        rt = ctypes.CDLL("libcudart.so.13")
    except OSError:
        pytest.skip("no shared CUDA runtime")
    dims, n = (12, 12, 12, 12), 16
    ctx = context(dims)
    ctx.set_integer_workspace(1, 0)
    Us = [dev(synth.su3_links(dims, 0.45, 40 + i)) for i in range(2)]
    xs = [field(dims, n, 50 + i) for i in range(2)]
    want = [ctx.wilson_apply(Us[i], KAPPA, xs[i]) for i in range(2)]
    outs = [torch.empty_like(xs[i % 2]) for i in range(6)]
    torch.cuda.synchronize()
    for i in range(6):
        s = ctypes.c_void_p()
        assert rt.cudaStreamCreateWithFlags(ctypes.byref(s), 1) == 0
        ctx.set_stream(s.value)
        ctx.wilson_apply(Us[i % 2], KAPPA, xs[i % 2], out=outs[i])
        assert rt.cudaStreamDestroy(s) == 0
    ctx.set_stream(torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    for i in range(6):
        assert torch.equal(outs[i], want[i % 2]), i
