"""The FP64 step in two passes (lbm_kernels_split.cuh), which tile kinds 5 and 6 take
with a launcher-chosen z chunk, against the pipelined kernel (kind 1): bitwise
equal fields for every stencil, tau = 1 and not, from the smallest boxes (blocks of
one warp) to ones with several warps a block, odd sides and partly empty last
blocks."""
import numpy as np
import pytest

import inputs
import paper_2105_08772_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box,stencil,tau", [
    ((3, 3, 3), "E4", 1.0), ((100, 3, 3), "E4", 1.0), ((37, 29, 23), "E4", 0.7), ((64, 56, 41), "E4", 1.0),
    ((5, 6, 5), "E6", 1.0), ((40, 20, 12), "E6", 1.3), ((5, 5, 7), "E8", 1.0), ((33, 17, 9), "E8", 0.8),
])
def test_two_passes_are_bitwise_the_pipelined_kernel(box, stencil, tau):
    f0 = inputs.random_populations(box[::-1], seed=sum(box))
    fields = []
    for other in (False, True):
        lat = P.Lattice(*box, tau=tau, G=-5.0, stencil=stencil, prec="f64")
        try:
            code = lat.get_tile()
            assert code // 10 ** 8 in (5, 6) and code // 10 % 1000 == 0, code
            if other:
                lat.set_tile(132040001)
            lat.set_populations(f0)
            lat.step(1)
            one = lat.get_populations()
            lat.step(6)
            fields.append((one, lat.get_populations()))
        finally:
            lat.close()
    for a, b in zip(*fields):
        assert np.isfinite(a).all() and np.array_equal(a, b)
