"""The register variants of the update, bit for bit, on lattices that fill the
GPU: smaller ones run a form of their own whatever the variant."""
import numpy as np
import pytest

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu

F12, F18 = su3.SU3_FP32_12, su3.SU3_FP32_18
KW = dict(beta=5.7, hits=2, start=su3.SU3_START_HOT, reunit_every=2)
# variant, threads, CTAs per SM: every variant at its largest CTA, at one warp, and on a persistent grid
SHAPES = [(v, t, c) for v, most in enumerate((256, 128, 128, 256, 256)) for t, c in ((most, 0), (32, 0), (64, 2))]

# more than 20 warps per SM of 152 are 97280 links of a phase
LATTICES = [
    ("torus", dict(dims=[24, 24, 24, 18], storage=F12)),                                   # 124416
    ("plain", dict(dims=[56, 60, 60], storage=F12)),                                       # 100800
    ("period", dict(dims=[24, 24, 24, 18], storage=F12, rng_period=[24, 24, 24, 6])),
    ("two-couplings", dict(dims=[20, 20, 16, 16], storage=F12, boundary=su3.SU3_DLT, beta1=4.8)),  # 102400
    ("torus-18", dict(dims=[24, 24, 24, 18], storage=F18)),
    ("two-couplings-18", dict(dims=[20, 20, 16, 16], storage=F18, boundary=su3.SU3_DLT, beta1=4.8)),
]


@pytest.mark.parametrize("name,kw", LATTICES, ids=[n for n, _ in LATTICES])
def test_lattice(name, kw):
    """Every variant and shape against the stage machine of a fused launch at
    variant 0."""
    cfgs = [su3.make_config(seed=s, **{**KW, **kw}) for s in (5, 6)]
    ens = su3.Ensemble(cfgs)
    ens.set_launch(128, 0, variant=0)
    ens.sweep(3)
    want = ens.get_links(0)
    ens.close()
    assert np.abs(want).max() < 1.1
    for variant, threads, ctas in SHAPES:
        if variant and kw["storage"] == F18:
            continue
        with su3.Lattice(seed=5, **{**KW, **kw}) as lat:
            lat.set_launch(threads, ctas, variant=variant)
            lat.sweep(3)
            assert np.array_equal(lat.get_links(), want), (variant, threads, ctas)


@pytest.mark.parametrize("kind", ["torus", "plain", "two-couplings"])
def test_ensemble(kind):
    """The fused launch in every variant and shape against each chain alone."""
    extra = {"torus": [], "plain": [dict(dims=[12, 14, 10])],
             "two-couplings": [dict(dims=[6, 8, 6, 4], boundary=su3.SU3_DLT, beta1=4.8)]}[kind]
    chains = [dict(dims=[8, 8, 8, 8])] * 3 + [dict(dims=[12, 12, 12, 12]), dict(dims=[6, 4, 10, 8])] + extra
    cfgs = [{**KW, "storage": F12, "seed": 30 + i, **c} for i, c in enumerate(chains)]
    want = []
    for c in cfgs:
        with su3.Lattice(**c) as lat:
            lat.sweep(3)
            want.append(lat.get_links())
    for variant, threads, ctas in SHAPES:
        ens = su3.Ensemble([su3.make_config(**c) for c in cfgs])
        ens.set_launch(threads, ctas, variant=variant)
        ens.sweep(3)
        for i, w in enumerate(want):
            assert np.array_equal(ens.get_links(i), w), (variant, threads, ctas, i)
        ens.close()


@pytest.mark.parametrize("storage", [F12, F18])
def test_divided_lattice(storage):
    """A divided lattice beyond the early form's 8 warps per SM (38912 links of
    a phase), in every launch shape, against the undivided one."""
    kw = dict(KW, dims=[18, 18, 18, 16], storage=storage, seed=7)  # 46656
    with su3.Lattice(**kw) as lat:
        lat.sweep(3)
        want = lat.get_links()
    for threads, ctas in ((256, 0), (32, 0), (64, 2), (128, 1)):
        with su3.Lattice(ndiv=(3, 1, 1, 2), **kw) as lat:
            lat.set_launch(threads, ctas)
            lat.sweep(3)
            assert np.array_equal(lat.get_links(), want), (threads, ctas)
