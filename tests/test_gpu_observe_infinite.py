"""Observables of a node whose density has overflowed: its velocity is the quotient
(j + F/2) / n, which is 0 for an infinite n and finite j + F/2, and the run is reported
as non-finite (status bit 3)."""
import numpy as np
import pytest

import inputs
import paper_2105_08772_gb300 as P

pytestmark = pytest.mark.gpu


def test_velocity_of_an_infinite_density_is_zero():
    box, at = (12, 9, 7), (3, 4, 5)      # node (z, y, x)
    f = inputs.random_populations(box[::-1], seed=3)
    f[(slice(1, 3),) + at] = 1.2e308     # an opposite pair: n = inf, j finite
    lat = P.Lattice(*box, G=-5.0, prec="f64")
    try:
        lat.set_populations(f)
        u = lat.velocity()
        assert np.isfinite(u).all()
        assert (u[(slice(None),) + at] == 0.0).all()
        o = lat.observables()
        assert (o.status_bits & 8) and np.isfinite(o.max_u) and np.isinf(o.mass)
    finally:
        lat.close()
