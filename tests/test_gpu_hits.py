"""su3_sweep with hits that change from call to call."""
import time

import numpy as np
import pytest

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu

KW = dict(beta=5.7, seed=6, storage=su3.SU3_FP32_12, start=su3.SU3_START_HOT, reunit_every=5, measure_every=2)


@pytest.mark.parametrize("dims", [[8, 8, 8, 4], [16, 16, 16, 8]], ids=str)
def test_changing_hits_equal_plain_launches(dims):
    """Six values in turn, more than there are sets of graphs, each several
    times: the links and counters are those of kernel by kernel launches."""
    got = []
    for graph in (True, False):
        with su3.Lattice(dims, **KW) as lat:
            lat.use_graph(graph)
            for i, hits in enumerate([1, 2, 1, 2, 3, 4, 5, 1, 6, 2, 6, 5, 4, 3, 2, 1, 1, 2]):
                lat.sweep(1 + i % 6, hits=hits)
            got.append((lat.get_links(), lat.stats()))
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]


def test_alternating_hits_capture_nothing_new():
    """A call that goes back to earlier hits takes its graph again.  Six values
    in turn are more than there are sets of graphs, so that every call captures:
    two values in turn cost the host well below that."""
    def host_time(lat, hits):
        t = []
        for k in range(48):
            lat.synchronize()
            t0 = time.perf_counter()
            lat.sweep(1, hits=hits[k % len(hits)])
            t.append(time.perf_counter() - t0)
        return np.median(t[12:])

    with su3.Lattice([8, 8, 8, 4], **dict(KW, measure_every=0)) as lat:
        two, six = host_time(lat, [1, 2]), host_time(lat, [1, 2, 3, 4, 5, 6])
    assert two < 0.6 * six, (two, six)
