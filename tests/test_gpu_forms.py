"""The update forms of one-chain engines (eight lanes per link, updates
begun before the previous launch has ended, parked draws, plain) against the stage machine
of a fused launch, bit for bit, on both sides of the lines between them."""
import numpy as np
import pytest

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu

F12, F18, F64 = su3.SU3_FP32_12, su3.SU3_FP32_18, su3.SU3_FP64_18
DLT = dict(boundary=su3.SU3_DLT)

CASES = [  # links of a phase (152 SMs)
    ("lanes-ragged", [6, 6, 10, 2], F12, {}),                    # 360
    ("lanes-D3", [14, 14, 12], F18, {}),                         # 1176
    ("lanes-dlt", [10, 6, 6, 4], F18, DLT),                      # 1440
    ("early-first", [16, 16, 10, 2], F12, {}),                    # 2560: one thread per link
    ("lanes-edge", [12, 12, 8, 4], F12, {}),                     # 2304
    ("early-D2", [128, 66], F12, {}),                            # 4224
    ("early-D3", [20, 18, 16], F18, {}),                         # 2880
    ("early-dlt", [16, 16, 14, 4], F12, dict(DLT, glue_mask=8)),  # 14336
    ("early-period", [10, 12, 10, 8], F12, dict(rng_period=[10, 12, 10, 4])),
    ("early-torus", [16, 16, 16, 10], F12, {}),                  # 20480: unrolled
    ("early-torus-18", [18, 18, 18, 12], F18, {}),               # 34992
    ("early-D3-two", [64, 32, 34], F12, {}),                     # 34816: rolled, two warps per scheduler
    ("parked-torus", [18, 18, 18, 14], F12, {}),                 # 40824
    ("parked-18", [20, 20, 20, 16], F18, {}),                    # 64000
    ("parked-period", [18, 18, 18, 18], F12, dict(rng_period=[18, 18, 18, 6])),  # 52488
    ("parked-dlt", [20, 20, 20, 10], F12, DLT),                  # 80000
    ("parked-last", [54, 60, 60], F12, {}),                      # 97200: 20 warps per SM are 97280 links
    ("plain-first", [56, 60, 60], F12, {}),                      # 100800
    ("plain-18", [20, 20, 20, 20], F18, {}),                     # 80000
    ("lanes-64-D3", [24, 20, 20], F64, {}),                      # 4800: lanes alone, not with a second chain
    ("plain-64-D2", [128, 78], F64, {}),                         # 4992
    ("plain-64-D3", [20, 20, 16], F64, DLT),                     # 6400
]


@pytest.mark.parametrize("name,dims,storage,kw", CASES, ids=[c[0] for c in CASES])
def test_forms_equal_the_stage_machine(name, dims, storage, kw):
    kw = dict(kw, dims=dims, storage=storage, beta=5.7 if len(dims) == 4 else 9.0, hits=2, start=su3.SU3_START_HOT,
              reunit_every=5)
    ens = su3.Ensemble([su3.make_config(seed=s, **kw) for s in (5, 6)])
    ens.sweep(14)
    want = ens.get_links(0)
    ens.close()
    # the default shape, short and long CTAs, a persistent grid of several tiles per CTA
    for shape in (None, (32, 0), (256, 0), (64, 1)):
        with su3.Lattice(seed=5, **kw) as lat:
            if shape:
                lat.set_launch(*shape, 0)
            for n in (1, 4, 9):
                lat.sweep(n)
            assert np.array_equal(lat.get_links(), want), shape


@pytest.mark.parametrize("dims,storage,ndiv,kw", [
    ([8, 8, 8, 4], F12, (2, 2, 1, 1), {}),                  # lanes
    ([12, 12, 12, 4], F12, (2, 1, 2, 1), {}),               # begun early
    ([12, 10, 12, 8], F18, (1, 5, 2, 2), {}),               # boxes two sites wide
    ([12, 12, 12, 4], F12, (2, 2, 1, 1), dict(DLT, glue_mask=8)),
    ([18, 18, 18, 12], F12, (3, 1, 1, 2), {}),              # two warps per scheduler
], ids=str)
def test_divided_forms_equal_the_undivided(dims, storage, ndiv, kw):
    kw = dict(kw, dims=dims, storage=storage, beta=5.7, hits=2, seed=8, start=su3.SU3_START_HOT, reunit_every=5)
    with su3.Lattice(**kw) as a, su3.Lattice(ndiv=ndiv, **kw) as b:
        for n in (1, 4, 9):
            a.sweep(n)
            b.sweep(n)
        assert np.array_equal(a.get_links(), b.get_links())
