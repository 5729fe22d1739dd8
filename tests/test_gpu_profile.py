"""Kernel timing counts a sweep's stages whatever launches run them."""
import pytest

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu


# a cluster's launch of whole sweeps, a launch per phase, and that of a divided lattice
@pytest.mark.parametrize("dims,ndiv", [([4, 4, 4, 4], None), ([8, 16], None), ([8, 8, 8, 4], None),
                                       ([4, 4, 4, 4], (2, 1, 1, 1))], ids=str)
@pytest.mark.parametrize("storage", [su3.SU3_FP32_12, su3.SU3_FP64_18])
def test_profile_counts_stages(dims, ndiv, storage):
    with su3.Lattice(dims, beta=5.7, storage=storage, start=su3.SU3_START_HOT, reunit_every=5, measure_every=4,
                     ndiv=ndiv) as lat:
        lat.set_profiling(True)
        lat.sweep(23)
        p = lat.profile(reset=True)
        assert (p["update_launches"], p["reunit_launches"], p["measure_launches"]) == (23 * 2 * len(dims), 4, 5)
        assert min(p["update_ms"], p["reunit_ms"], p["measure_ms"]) > 0.0
        assert lat.profile()["update_launches"] == 0
