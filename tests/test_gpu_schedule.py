"""A lattice's fixed schedule (one kernel per stage, graphs of whole sweeps)
against the stage machine of a fused launch, bit for bit."""
import numpy as np
import pytest

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu

CASES = [
    dict(dims=[4, 4, 4, 4], storage=su3.SU3_FP32_12),
    dict(dims=[6, 10], storage=su3.SU3_FP32_18),
    dict(dims=[6, 4, 8], storage=su3.SU3_FP32_12),
    dict(dims=[4, 6, 4, 2], storage=su3.SU3_FP64_18),
    dict(dims=[4, 4, 2, 4], storage=su3.SU3_FP32_12, boundary=su3.SU3_DLT),
]


@pytest.mark.parametrize("kw", CASES, ids=lambda k: "x".join(map(str, k["dims"])))
@pytest.mark.parametrize("reunit,measure", [(0, 0), (3, 2), (1, 1), (5, 0), (0, 7)])
def test_pieces_equal_the_stage_machine(kw, reunit, measure):
    """23 sweeps in pieces that end before, at and after every cadence."""
    kw = dict(kw, beta=5.7, hits=2, start=su3.SU3_START_HOT, reunit_every=reunit, measure_every=measure)
    ens = su3.Ensemble([su3.make_config(seed=s, **kw) for s in (5, 6)])
    ens.sweep(23)
    want, wm = ens.get_links(0), ens.measurements(0)
    ens.close()
    for graph in (True, False):
        with su3.Lattice(seed=5, **kw) as lat:
            lat.use_graph(graph)
            for n in (1, 2, 3, 4, 5, 0, 8):
                lat.sweep(n)
            assert np.array_equal(lat.get_links(), want)
            m = lat.measurements()
            assert m.shape == wm.shape
            # the two forms sum the sites in different orders
            assert np.allclose(m, wm, rtol=0, atol=1e-14)
            assert lat.stats()[2] == 23
