"""Sweeps queued on a caller's stream while the caller captures it."""
import numpy as np
import pytest
import torch

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,storage", [([4, 4, 4, 4], su3.SU3_FP64_18), ([8, 8, 8, 4], su3.SU3_FP32_12),
                                          ([16, 16, 16, 8], su3.SU3_FP32_18)], ids=str)
def test_sweeps_in_a_captured_stream(dims, storage):
    """The sweeps become part of the caller's graph (they are launched kernel
    by kernel there), and run when it is replayed."""
    kw = dict(beta=5.7, seed=11, storage=storage, start=su3.SU3_START_HOT, hits=2, reunit_every=4, measure_every=2)
    stream = torch.cuda.Stream()
    with su3.Lattice(dims, stream=stream, **kw) as lat, su3.Lattice(dims, **kw) as ref:
        lat.sweep(4)  # every kernel is loaded
        lat.synchronize()
        before = lat.get_links()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            lat.sweep(1)
            lat.sweep(3)
        torch.cuda.synchronize()
        assert np.array_equal(lat.get_links(), before)  # nothing has run yet
        with torch.cuda.stream(stream):
            graph.replay()
        lat.sweep(2)
        ref.sweep(10)
        assert np.array_equal(lat.get_links(), ref.get_links())
        assert lat.stats() == ref.stats()
        assert np.array_equal(lat.measurements(), ref.measurements())
        del graph
