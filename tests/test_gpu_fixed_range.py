"""FP64 links outside the range of the fixed-point update: the sites they
reach are updated by the double-precision form, which a fused launch takes
for all chains when one of them has two couplings."""
import numpy as np
import pytest
import torch

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu

TWO = dict(dims=[4, 2, 2, 2], boundary=su3.SU3_DLT, beta=5.0, beta1=4.0)
# a cluster's launch, eight lanes per link (with a ragged tile), one thread per link, divided
SHAPES = [([4, 4, 4, 4], None), ([6, 10, 8, 6], None), ([16, 16, 16, 8], None), ([16, 16, 16, 8], (2, 1, 1, 2))]


def rotated(dims, scale, seed):
    """Links scale * g(x) g(x + mu)^+ with random SU(3) matrices g, canonical layout."""
    rng = np.random.default_rng(seed)
    z = rng.standard_normal((*dims[::-1], 3, 3, 2))
    g, _ = np.linalg.qr(z[..., 0] + 1j * z[..., 1])
    g = g / np.linalg.det(g)[..., None, None] ** (1 / 3)
    D = len(dims)
    U = np.stack([scale * g @ np.conj(np.swapaxes(np.roll(g, -1, axis=D - 1 - mu), -1, -2)) for mu in range(D)], axis=D)
    return np.stack([U.real, U.imag], axis=-1).reshape(1, -1, D, 3, 3, 2)


def first_phase(links, dims):
    """The links of colour 0 in direction 0: no later phase of the sweep changes them."""
    x = np.indices(dims[::-1]).sum(axis=0).reshape(-1)
    return links[0, x % 2 == 0, 0].reshape(-1, 18)


def double_form(dims, links, **kw):
    """One sweep of the double-precision form."""
    buf = torch.zeros(links.size, device="cuda", dtype=torch.float64)
    with su3.Lattice(dims, buffer=buf, **kw) as lat:
        lat.set_links(links)
        start = buf.clone()
    ens = su3.Ensemble([su3.make_config(dims, buffer=buf, **kw), su3.make_config(**TWO)])
    ens.sweep(0)
    ens.get_links(0)  # the start configuration is written
    buf.copy_(start)
    torch.cuda.synchronize()
    ens.sweep(1)
    out = ens.get_links(0)
    ens.close()
    return out


@pytest.mark.parametrize("scale", [1.05, 1.07])
@pytest.mark.parametrize("dims,ndiv", SHAPES, ids=str)
def test_scaled_links(dims, ndiv, scale):
    """Links off SU(3) by a few per cent whose elements and products all pass
    the range check: the projections reach 6 x 1.07^4 = 7.9 on average and 8
    on many sites.  Every link stays within the parity bound."""
    start = rotated(dims, scale, 3)
    kw = dict(beta=6.0, hits=2, seed=21)
    want = first_phase(double_form(dims, start, **kw), dims)
    with su3.Lattice(dims, ndiv=ndiv, **kw) as lat:
        lat.set_links(start)
        lat.sweep(1)
        got = first_phase(lat.get_links(), dims)
    assert np.abs(want - first_phase(start, dims)).max() > 0.1  # the update did move them
    assert np.max(np.abs(got - want)) <= 1e-11
