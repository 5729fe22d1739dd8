"""FP64 links outside the range of the fixed-point update: the sites they
reach are updated by the double-precision form, which chains of two couplings
take for every site."""
import numpy as np
import pytest

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu

# a cluster's launch, eight lanes per link (with a ragged tile), one thread per
# link, and that of a divided lattice; each of the two layers
SHAPES = [([4, 4, 4, 2], None), ([6, 10, 8, 6], None), ([16, 16, 16, 4], None), ([16, 16, 16, 4], (2, 1, 2, 1))]
DLT = dict(boundary=su3.SU3_DLT, glue_mask=8)  # glued in time


def rotated(dims, scale, seed):
    """Links scale * g(x) g(x + mu)^+ with random SU(3) matrices g on the double
    layer (a step across the time boundary lands in the other one), canonical
    layout."""
    rng = np.random.default_rng(seed)
    z = rng.standard_normal((2, *dims[::-1], 3, 3, 2))
    g, _ = np.linalg.qr(z[..., 0] + 1j * z[..., 1])
    g = g / np.linalg.det(g)[..., None, None] ** (1 / 3)
    D = len(dims)
    U = []
    for mu in range(D):
        far = np.roll(g, -1, axis=D - mu)
        if mu == D - 1:
            far[:, -1] = far[::-1, -1].copy()
        U.append(scale * g @ np.conj(np.swapaxes(far, -1, -2)))
    U = np.stack(U, axis=D + 1)
    return np.stack([U.real, U.imag], axis=-1).reshape(2, -1, D, 3, 3, 2)


def first_phase(links, dims):
    """The links of colour 0 in direction 0: no later phase of the sweep changes them."""
    x = np.indices(dims[::-1]).sum(axis=0).reshape(-1)
    return links[:, x % 2 == 0, 0].reshape(-1, 18)


def one_sweep(dims, links, beta, **kw):
    with su3.Lattice(dims, beta=beta, hits=2, seed=21, **DLT, **kw) as lat:
        lat.set_links(links)
        lat.sweep(1)
        return lat.get_links()


def double_form(dims, links, beta):
    """One sweep of the double-precision form: the second coupling is the next
    double above the first."""
    return one_sweep(dims, links, beta, beta1=float(np.nextafter(beta, 10.0)))


@pytest.mark.parametrize("scale", [1.05, 1.07])
@pytest.mark.parametrize("dims,ndiv", SHAPES, ids=str)
def test_scaled_links(dims, ndiv, scale):
    """Links off SU(3) by a few per cent whose elements and products all pass
    the range check: the projections reach 6 x 1.07^4 = 7.9 on average and 8
    on many sites.  Every link stays within the parity bound."""
    start = rotated(dims, scale, 3)
    want = first_phase(double_form(dims, start, 6.0), dims)
    got = first_phase(one_sweep(dims, start, 6.0, ndiv=ndiv), dims)
    assert np.abs(want - first_phase(start, dims)).max() > 0.1  # the update did move them
    assert np.max(np.abs(got - want)) <= 1e-11


def bad_link_case(dims, seed):
    """A bad link of layer 0 in each place of a first-phase update: the link
    itself (direction 0, colour 0), a staple's parallel link (direction 0,
    colour 1) and its side links (direction 1, either colour).  Its site, its
    direction and the sites of the links that it enters as (layer, site)."""
    x = np.indices(dims[::-1]).reshape(len(dims), -1)[::-1].T  # x[site] = coordinates, x^1 fastest
    colour = x.sum(axis=1) % 2
    e = np.eye(len(dims), dtype=int)

    def place(c):  # the time direction is glued
        layer = int(c[-1] // dims[-1]) % 2
        c = [int(k) % n for k, n in zip(c, dims)]
        return layer, int(np.ravel_multi_index(c[::-1], dims[::-1]))

    rng = np.random.default_rng(seed)
    for mu, col in ((0, 0), (0, 1), (1, 0), (1, 1)):
        y = x[rng.choice(np.flatnonzero(colour == col))]
        if mu == 0:  # U_0(y), and the links whose staples hold it: y +- nu
            near = [y] if col == 0 else [y + s * e[nu] for nu in range(1, len(dims)) for s in (1, -1)]
        else:        # U_1(y) stands beside U_0 at y, y + 1, y - 0 and y - 0 + 1
            near = [y, y + e[1], y - e[0], y - e[0] + e[1]]
        yield place(y)[1], mu, sorted({place(c) for c in near if sum(c) % 2 == 0})


@pytest.mark.parametrize("dims,ndiv", SHAPES, ids=str)
@pytest.mark.parametrize("bad", [1.5, -1.2, 40.0])
def test_sites_of_one_bad_link(dims, ndiv, bad):
    """One element out of range: of the links of the first phase those that the
    bad link enters are the double form's within the parity bound, and all
    others are the bits they have without it."""
    with su3.Lattice(dims, beta=5.7, seed=9, start=su3.SU3_START_HOT, **DLT) as lat:
        good = lat.get_links()
    without = one_sweep(dims, good, 5.7, ndiv=ndiv)[:, :, 0]
    first = np.indices(dims[::-1]).sum(axis=0).reshape(-1) % 2 == 0
    for y, mu, near in bad_link_case(dims, 4):
        links = good.copy()
        links[0, y, mu, 1, 2, 0] = bad
        got, double = (f[:, :, 0] for f in (one_sweep(dims, links, 5.7, ndiv=ndiv), double_form(dims, links, 5.7)))
        touched = np.zeros((2, len(first)), dtype=bool)
        touched[tuple(zip(*near))] = True
        assert np.abs(got[touched] - double[touched]).max() <= 1e-11 * max(1.0, abs(bad)), (mu, y)
        far = first & ~touched
        assert np.array_equal(got[far], without[far]), (mu, y)
        assert not np.array_equal(double[far], without[far])  # the two forms do differ in their last bits
