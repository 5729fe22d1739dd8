"""The job server's device memory."""
import time

import numpy as np
import pytest
import torch

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu


@pytest.fixture
def disarm():
    yield
    su3.su3_inject_fault("server_pool", 0)


def config(dims, seed=3, **kw):
    return su3.make_config(dims, beta=5.7, seed=seed, storage=su3.SU3_FP32_12, start=su3.SU3_START_HOT, hits=2,
                           reunit_every=10, **kw)


def test_jobs_run_without_a_pool(disarm):
    """Where no memory pool can be made the jobs' memory comes from plain
    allocations, and links go in and out as ever."""
    dims, links = [8, 8, 8, 4], []
    su3.su3_inject_fault("server_pool", 1)
    srv = su3.Server(max_slots=2)
    for n in (5, 7):  # the second job starts from the first one's links
        out = np.zeros((1, 8 * 8 * 8 * 4, 4, 3, 3, 2))
        job = srv.submit(config(dims), n, links_in=links[-1] if links else None, links_out=out)
        assert srv.wait(job, timeout_s=60).status == su3.SU3_OK
        links.append(out)
    srv.close()
    with su3.Lattice(dims, beta=5.7, seed=3, storage=su3.SU3_FP32_12, start=su3.SU3_START_HOT, hits=2,
                     reunit_every=10) as lat:
        for n, out in zip((5, 7), links):
            lat.set_sweep_counter(0)
            lat.sweep(n)
            assert np.array_equal(lat.get_links(), out)


def test_idle_server_gives_its_memory_back():
    """A 32^4 job holds 201 MB of links; a server that has been idle for a
    while keeps 32 MiB at most."""
    dims = [32, 32, 32, 32]
    size = su3.su3_link_bytes(config(dims))
    srv = su3.Server(max_slots=2)
    # what the first job brings once: the context, modules, the worker's buffers
    assert srv.wait(srv.submit(config([4, 4, 4, 4]), 1), timeout_s=60).status == su3.SU3_OK
    before = torch.cuda.mem_get_info()[0]
    assert srv.wait(srv.submit(config(dims), 1), timeout_s=60).status == su3.SU3_OK
    deadline = time.time() + 10
    while torch.cuda.mem_get_info()[0] < before - size // 4 and time.time() < deadline:
        time.sleep(0.05)
    assert torch.cuda.mem_get_info()[0] >= before - size // 4
    # and takes jobs as before
    assert srv.wait(srv.submit(config(dims), 1), timeout_s=60).status == su3.SU3_OK
    srv.close()


@pytest.mark.parametrize("dims,layers", [([4, 4, 4, 4], 1), ([8, 8, 8, 4], 2), ([24, 24, 24], 1)], ids=str)
def test_budget_of_one_job(dims, layers):
    """A job needs its links, 32 bytes of partial sums and 8 of booked action
    per 32 sites of a colour, its ring of measurements and two counters: a
    budget of that takes it, one byte less does not."""
    cfg = config(dims, boundary=su3.SU3_DLT if layers == 2 else su3.SU3_PBC, measure_every=2, measure_capacity=16)
    tiles = layers * -(-int(np.prod(dims)) // 64)
    need = su3.su3_link_bytes(cfg) + tiles * 40 + 16 * (layers + 1) * 40 + 16
    srv = su3.Server(hbm_budget_bytes=need, max_slots=2)
    assert srv.wait(srv.submit(cfg, 4), timeout_s=60).status == su3.SU3_OK
    srv.close()
    srv = su3.Server(hbm_budget_bytes=need - 1, max_slots=2)
    with pytest.raises(su3.Su3Error) as ei:
        srv.submit(cfg, 4)
    assert ei.value.status == su3.SU3_ENOMEM
    srv.close()
