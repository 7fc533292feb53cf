"""Groups on the row kernel: uneven boxes of one launch evolve bitwise as under
lbm_step -- aligned boxes, a mix of aligned and odd ones, several rounds of items,
odd step counts (the table's parities), FP32.  Boxes from three rows an item to
many, so that an item's last density and collision pieces are partly empty."""
import numpy as np
import pytest

import paper_2105_08772_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("boxes", [
    [(64, 64, 64), (72, 40, 33), (96, 24, 50)],                   # aligned rows
    [(61, 60, 43), (64, 64, 40), (335, 9, 12), (33, 47, 29)],     # any rows
    [(128, 128, 96), (112, 112, 112), (80, 80, 80)],              # several rounds
])
def test_group_on_the_row_kernel_is_bitwise_single(boxes):
    lats, refs = [], []
    try:
        for k, box in enumerate(boxes):
            for out in (lats, refs):
                lat = P.Lattice(*box, G=-5.0, prec="f32")
                lat.init_drop([n // 2 for n in box], min(box) / 4.0, 1.9 - 0.1 * k, 0.13)
                out.append(lat)
        g = P.Group(lats)
        for n in (1, 6, 130):
            g.step(n)
            for lat in refs:
                lat.step(n)
        for a, b in zip(lats, refs):
            pa, pb = a.get_populations(), b.get_populations()
            assert np.isfinite(pa).all() and np.array_equal(pa, pb)
            assert a.observables().steps == 137 and not (a.observables().status_bits & 16)
        g.close()
    finally:
        for lat in lats + refs:
            lat.close()
