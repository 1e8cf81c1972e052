"""Entries at the ends of the FP64 range, and far apart within a site, through the kernels that run on integers."""
import numpy as np
import pytest

from oracle import lattice as L, operators as O
from paper_1903_06986_gb300 import synth
from tests.gpu_util import context, dev, rel_err

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
