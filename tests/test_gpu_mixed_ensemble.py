"""Chains beside chains of two couplings in one fused launch."""
import numpy as np
import pytest

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu

CHAINS = [
    dict(dims=[8, 8, 8, 8]),
    dict(dims=[6, 4, 10, 8], boundary=su3.SU3_DLT),
    dict(dims=[4, 4, 6, 4], boundary=su3.SU3_DLT, beta1=4.5),
    dict(dims=[10, 12, 6]),
    dict(dims=[6, 6, 4, 4], boundary=su3.SU3_DLT, glue_mask=8, beta1=7.0),
]


@pytest.mark.parametrize("storage", [su3.SU3_FP64_18, su3.SU3_FP32_12, su3.SU3_FP32_18])
def test_every_chain_equals_itself_alone(storage):
    """Links, measurements and couplings do not mix: each chain gives the bits
    that it gives alone, one coupling or two."""
    cfgs = [dict(beta=5.7, hits=2, storage=storage, seed=60 + i, start=su3.SU3_START_HOT, reunit_every=3, **c)
            for i, c in enumerate(CHAINS)]
    for shape in ((128, 0), (64, 2)):
        ens = su3.Ensemble([su3.make_config(**c) for c in cfgs])
        ens.set_launch(*shape)
        ens.sweep(5)
        for i, c in enumerate(cfgs):
            with su3.Lattice(**c) as lat:
                lat.sweep(5)
                assert np.array_equal(ens.get_links(i), lat.get_links()), (shape, c)
        ens.close()
