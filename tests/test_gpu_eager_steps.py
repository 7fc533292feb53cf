"""Steps launched one by one and steps replayed from a graph take different kernels in
small FP32 boxes; the fields are bitwise equal, on both sides of the line."""
import numpy as np
import pytest

import inputs
import paper_2105_08772_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box,stencil,tau", [
    ((8, 8, 8), "E4", 1.0), ((32, 32, 32), "E4", 1.0), ((33, 33, 33), "E4", 1.0), ((100, 3, 3), "E4", 0.8),
    ((48, 40, 12), "E4", 1.0), ((48, 40, 12), "E4", 1.3), ((100, 5, 5), "E6", 1.0), ((67, 5, 6), "E8", 0.8),
])
def test_eager_and_replayed_steps_agree(box, stencil, tau):
    f0 = inputs.random_populations(box[::-1], seed=sum(box))
    fields = []
    for calls in ([128] * 2, [1] * 4 + [63, 61] + [64] * 2):
        lat = P.Lattice(*box, tau=tau, G=-5.0, stencil=stencil, prec="f32")
        try:
            lat.set_populations(f0)
            for n in calls:
                lat.step(n)
            fields.append(lat.get_populations())
        finally:
            lat.close()
    assert np.isfinite(fields[0]).all() and np.array_equal(*fields)
