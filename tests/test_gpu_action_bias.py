"""The booked action of FP64 chains has no one-sided error."""
import pytest

import paper_0904_0642_gb300 as su3

pytestmark = pytest.mark.gpu


# a cluster's launch, eight lanes per link, one thread per link, and that of a divided lattice
@pytest.mark.parametrize("dims,ndiv,sweeps", [([4, 4, 4, 4], None, 2000), ([8, 8, 8, 8], None, 200),
                                              ([16, 16, 16, 8], None, 200), ([16, 16, 16, 8], (2, 1, 1, 2), 200)],
                         ids=str)
def test_mean_booking_error(dims, ndiv, sweeps):
    """One update's change of Re Tr(U A) is of size 1 to 12, and its rounding
    must not add up: over many updates the booked and the direct action differ
    by less than 2^-53 of Re Tr per update, on average, plus the rounding of
    the two sums (8 x 2^-53 of the action)."""
    beta = 6.0
    with su3.Lattice(dims, beta=beta, seed=9, storage=su3.SU3_FP64_18, start=su3.SU3_START_HOT, ndiv=ndiv) as lat:
        lat.sweep(20)
        lat.reunitarize()
        lat.action_reset()
        lat.sweep(sweeps)
        booked, direct = lat.action()
        bound = 2.0 ** -53 * beta / 3 * lat.nlinks * sweeps + 8 * 2.0 ** -53 * direct
    assert abs(booked - direct) <= bound, ((booked - direct) / bound, bound)
