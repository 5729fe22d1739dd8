"""The fixed-point forms of the FP64 update: eight lanes per link and one
thread per link give the same bits, and links outside the fixed-point range
take the double-precision form."""
import numpy as np
import pytest
import torch

import oracle
import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu

# few links (eight lanes per link) in every geometry; ragged tiles among them
SHAPES = [
    dict(dims=[4, 4, 4, 4]),
    dict(dims=[6, 4, 2, 10]),
    dict(dims=[2, 2, 2, 2]),
    dict(dims=[10, 6]),
    dict(dims=[6, 4, 14]),
    dict(dims=[4, 2, 4, 4], boundary=su3.SU3_DLT),
    dict(dims=[4, 4, 2, 4], boundary=su3.SU3_DLT, glue_mask=0b1000),
]
BIG = dict(dims=[16, 16, 16, 8])  # 16384 links per phase: with it an ensemble runs one thread per link


@pytest.mark.parametrize("beta,hits", [(5.7, 2), (0.6, 3), (60.0, 1), (0.0, 2)])
def test_forms_agree_bitwise(beta, hits):
    cfgs = [su3.make_config(seed=40 + i, beta=beta, hits=hits, start=su3.SU3_START_HOT, reunit_every=2, **s)
            for i, s in enumerate(SHAPES + [BIG])]
    ens = su3.Ensemble(cfgs)
    ens.sweep(3)
    for i, s in enumerate(SHAPES):
        with su3.Lattice(seed=40 + i, beta=beta, hits=hits, start=su3.SU3_START_HOT, reunit_every=2, **s) as lat:
            lat.sweep(3)
            assert np.array_equal(lat.get_links(), ens.get_links(i)), s
    ens.close()


@pytest.mark.parametrize("dims", [[4, 4, 4, 4], [16, 16, 16, 8]])
@pytest.mark.parametrize("bad", [1.5, np.inf, np.nan])
def test_links_out_of_range(dims, bad):
    """One link scaled out of range: every link whose staple it enters, and the
    link itself, must be the double-precision form's (a two-coupling chain in
    the same ensemble selects it for all), bit for bit in the first phase;
    links away from it stay within the parity bound."""
    two = su3.make_config([4, 2, 2, 2], boundary=su3.SU3_DLT, beta=5.0, beta1=4.0)
    got = []
    for extra in ([], [two]):
        buf = torch.zeros(int(np.prod(dims)) * 4 * 18, device="cuda", dtype=torch.float64)
        ens = su3.Ensemble([su3.make_config(dims, beta=5.7, seed=9, start=su3.SU3_START_HOT, buffer=buf)] + extra)
        torch.cuda.synchronize()
        # the first real part of a colour-1 link in direction 0 (first plane group of colour 1)
        vh = int(np.prod(dims)) // 2
        at = (4 * 9 * vh + vh // 3) * 2
        buf[at] = bad if not np.isfinite(bad) else buf[at] + bad
        ens.sweep(1)
        got.append(ens.get_links(0))
        ens.close()
    a, b = (x.reshape(-1, 18) for x in got)
    nan = np.isnan(b).any(axis=1)
    assert np.array_equal(nan, np.isnan(a).any(axis=1))
    if not np.isfinite(bad):
        assert nan.any()
    same = np.abs(a[~nan] - b[~nan])
    # a scaled link makes badly conditioned neighbours; the rest of the lattice is unaffected
    assert np.median(same.max(axis=1)) < 1e-12 and (same.max(axis=1) < 1e-8).mean() > 0.99


def test_cold_start_and_small_elements():
    """Zeros, and elements of every size down to the smallest doubles."""
    o = oracle.Lattice([4, 4, 4, 4]).cold_start()
    rng = np.random.default_rng(1)
    for mag in (0.0, 1e-3, 1e-9, 1e-15, 1e-300):
        U = oracle.Lattice([4, 4, 4, 4]).cold_start().U + mag * rng.standard_normal(o.U.shape)
        w = oracle.Lattice([4, 4, 4, 4])
        w.U[...] = U
        w.reunitarize()
        U = w.U.copy()
        w.sweep(6.0, 2, 3, n=1)
        with su3.Lattice([4, 4, 4, 4], beta=6.0, seed=3, hits=2) as lat:
            lat.set_links(U)
            lat.sweep(1)
            assert np.max(np.abs(lat.get_links() - w.U)) <= 1e-11, mag
