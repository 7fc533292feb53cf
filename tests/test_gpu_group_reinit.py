"""A group whose lattices are initialised again: the new storage shift reaches the
group's next steps, so that it still evolves bitwise as separate lattices do.  A
fresh drop starts with the same buffer parity as before, so the parity alone does
not show the change; other densities give another mean, hence another shift."""
import numpy as np
import pytest

import inputs
import paper_2105_08772_gb300 as P

pytestmark = pytest.mark.gpu

BOXES = [(48, 40, 36), (37, 29, 23)]


@pytest.mark.parametrize("steps", [6, 130])     # plain launches, graph replays
@pytest.mark.parametrize("how", ["init_drop", "init_rho", "set_populations"])
def test_group_follows_a_new_initial_field(how, steps):
    grouped = [P.Lattice(*b, G=-5.0, prec="f32") for b in BOXES]
    alone = [P.Lattice(*b, G=-5.0, prec="f32") for b in BOXES]
    try:
        for lat, box in zip(grouped, BOXES):
            lat.init_drop([n // 2 for n in box], 6.0, 1.89, 0.12)
        g = P.Group(grouped)
        g.step(steps)
        for lats in (grouped, alone):
            for k, (lat, box) in enumerate(zip(lats, BOXES)):
                f = inputs.random_populations(box[::-1], seed=5 + k)
                if how == "init_drop":
                    lat.init_drop([n // 2 for n in box], 9.0, 0.2, 1.7)
                elif how == "init_rho":
                    lat.init_rho(f.sum(axis=0))
                else:
                    lat.set_populations(f)
        g.step(steps)
        for a, b in zip(grouped, alone):
            b.step(steps)
            pa, pb = a.get_populations(), b.get_populations()
            assert np.isfinite(pa).all() and np.array_equal(pa, pb)
        g.close()
    finally:
        for lat in grouped + alone:
            lat.close()
