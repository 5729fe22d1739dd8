"""A driver that refuses programmatic launches: every call goes over to
ordinary ones, with the same results."""
import numpy as np
import pytest

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ndiv", [None, (2, 1, 1, 1)], ids=str)
@pytest.mark.parametrize("call", ["reunitarize", "sweep"])
def test_refused_launch_falls_back(call, ndiv):
    got = []
    for refused in (False, True):
        with su3.Lattice([8, 8, 8, 4], beta=5.7, seed=4, storage=su3.SU3_FP32_12, start=su3.SU3_START_HOT, hits=2,
                         ndiv=ndiv) as lat:
            lat.use_graph(False)
            lat.sweep(3)
            try:
                if refused:
                    su3.su3_inject_fault("programmatic", 1)
                lat.reunitarize() if call == "reunitarize" else lat.sweep(1)
            finally:
                su3.su3_inject_fault("programmatic", 0)
            lat.sweep(2)
            got.append(lat.get_links())
    assert np.array_equal(*got)
