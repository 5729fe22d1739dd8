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


def bad_link_case(dims, seed):
    """A bad link in each place of a first-phase update: the link itself
    (direction 0, colour 0), a staple's parallel link (direction 0, colour 1)
    and its side links (direction 1, either colour)."""
    V = int(np.prod(dims))
    x = np.indices(dims[::-1]).reshape(len(dims), -1)[::-1].T  # x[site] = coordinates, x^1 fastest
    colour = x.sum(axis=1) % 2
    site = lambda c: int(np.ravel_multi_index(tuple(int(k) % n for k, n in zip(c, dims))[::-1], dims[::-1]))
    rng = np.random.default_rng(seed)
    e = np.eye(len(dims), dtype=int)
    for mu, col in ((0, 0), (0, 1), (1, 0), (1, 1)):
        y = x[rng.choice(np.flatnonzero(colour == col))]
        if mu == 0:  # U_0(y), and the links whose staples hold it: y +- nu
            near = [y] if col == 0 else [y + s * e[nu] for nu in range(1, len(dims)) for s in (1, -1)]
        else:        # U_1(y) stands beside U_0 at y, y + 1, y - 0 and y - 0 + 1
            near = [y, y + e[1], y - e[0], y - e[0] + e[1]]
        near = sorted({site(c) for c in near if sum(c) % 2 == 0})
        yield site(y), mu, near, V


@pytest.mark.parametrize("dims,ndiv", SHAPES, ids=str)
@pytest.mark.parametrize("bad", [1.5, -1.2, 40.0])
def test_sites_of_one_bad_link(dims, ndiv, bad):
    """One element out of range: of the links of the first phase those that the
    bad link enters are the double form's bits, all others are the bits they
    have without it."""
    kw = dict(beta=5.7, hits=2, seed=9)
    with su3.Lattice(dims, start=su3.SU3_START_HOT, **kw) as lat:
        lat.reunitarize()
        good = lat.get_links()

    def swept(links):
        with su3.Lattice(dims, ndiv=ndiv, **kw) as lat:
            lat.set_links(links)
            lat.sweep(1)
            return lat.get_links()[0, :, 0]

    without = swept(good)
    first = np.flatnonzero(np.indices(dims[::-1]).sum(axis=0).reshape(-1) % 2 == 0)
    for y, mu, near, V in bad_link_case(dims, 4):
        links = good.copy()
        links[0, y, mu, 1, 2, 0] = bad
        got, double = swept(links), double_form(dims, links, **kw)[0, :, 0]
        assert np.array_equal(got[near], double[near]), (mu, y)
        far = np.setdiff1d(first, near)
        assert np.array_equal(got[far], without[far]), (mu, y)
        assert not np.array_equal(double[far], without[far])  # the two forms do differ in their last bits
