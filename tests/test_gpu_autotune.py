"""The autotuner reports a variant only where variants are different kernels."""
import numpy as np
import pytest

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu

ONE_KERNEL = [
    dict(dims=[4, 4, 4, 4]),                                          # whole sweeps per launch
    dict(dims=[8, 8, 8, 4]),                                          # eight lanes per link
    dict(dims=[16, 16, 16, 4], boundary=su3.SU3_DLT, glue_mask=8),    # begun early, rolled
    dict(dims=[16, 16, 16, 16]),                                      # begun early
    dict(dims=[12, 12, 12, 4], ndiv=(2, 1, 2, 1)),
]


@pytest.mark.parametrize("kw", ONE_KERNEL, ids=lambda k: "x".join(map(str, k["dims"])))
def test_one_kernel_has_variant_0(kw):
    with su3.Lattice(beta=6.0, seed=4, storage=su3.SU3_FP32_12, start=su3.SU3_START_HOT, hits=2, **kw) as lat:
        variant, threads, ctas, us = lat.autotune()
        assert variant == 0 and us > 0.0
        if kw["dims"] == [4, 4, 4, 4]:  # and its launch one shape
            assert (threads, ctas) == (128, 0)


def test_parked_draws_have_variant_0():
    """One CTA per tile runs the parked form whatever the variant; a
    persistent grid the variant itself.  The links do not depend on it."""
    kw = dict(beta=6.0, seed=4, storage=su3.SU3_FP32_12, start=su3.SU3_START_HOT, hits=2)
    with su3.Lattice([18, 18, 18, 14], **kw) as lat, su3.Lattice([18, 18, 18, 14], **kw) as ref:
        variant, _, ctas, _ = lat.autotune()
        assert variant == 0 or ctas > 0
        lat.sweep(2)
        ref.sweep(2)
        assert np.array_equal(lat.get_links(), ref.get_links())
