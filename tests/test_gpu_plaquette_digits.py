"""The FP64 plaquette keeps the digits of a double."""
import numpy as np
import pytest
import torch

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu


def random_su3(rng):
    q, _ = np.linalg.qr(rng.standard_normal((3, 3)) + 1j * rng.standard_normal((3, 3)))
    return q / np.linalg.det(q) ** (1 / 3)


def exact(V, W):
    """Re Tr(V W (W V)^+) in extended precision, third rows from rows 1, 2."""
    V, W = V.astype(np.clongdouble), W.astype(np.clongdouble)
    P, Q = V[:2] @ W, W[:2] @ V
    G = P.conj() @ Q.T
    return (G[0, 0] + G[1, 1] + G[0, 0] * G[1, 1] - G[0, 1] * G[1, 0]).real


@pytest.mark.parametrize("route", ["lattice", "noalloc"])
def test_constant_field(route):
    """A 4^2 lattice of constant links V, W: all plaquettes are equal, so the
    rounding of one does not average out.  Of Re Tr, of size 1: one rounding
    to a double (2^-53 at most), sums of sixteen equal values, and the division
    (2^-53) make less than 2^-51, root mean square over 64 fields."""
    rng = np.random.default_rng(8)
    buf = torch.zeros(4 * 4 * 2 * 18, device="cuda", dtype=torch.float64)
    out = torch.zeros(10, device="cuda", dtype=torch.float64)
    err = []
    with su3.Lattice([4, 4], buffer=buf) as lat:
        for _ in range(64):
            V, W = random_su3(rng), random_su3(rng)
            U = np.broadcast_to(np.stack([V, W]), (1, 16, 2, 3, 3))
            lat.set_links(np.ascontiguousarray(np.stack([U.real, U.imag], axis=-1)))
            if route == "lattice":
                p = lat.plaquette()[0]
            else:
                su3.su3_measure_noalloc(lat.cfg, buf.data_ptr(), out.data_ptr())
                torch.cuda.synchronize()
                p = float(out[0])
            err.append(float(3 * np.longdouble(p) - exact(V, W)))
    assert np.sqrt(np.mean(np.square(err))) < 2.0 ** -51
