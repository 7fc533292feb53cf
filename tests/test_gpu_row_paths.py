"""The row kernel on the boxes it is chosen for, by its plan (asserted, not assumed):
blocks that wrap in y once and on both sides, items of one row, one and several rounds
of items, partly empty last blocks and chunks; and groups with aligned and any rows.
Bitwise against the tile kernels, which a fixed z chunk selects."""
import numpy as np
import pytest

import launch_rules
import paper_2105_08772_gb300 as P

pytestmark = pytest.mark.gpu

ROW, ROW_ANY = 4, 5


def field(box):
    rng = np.random.default_rng(sum(box))
    rho = 1.0 + 0.6 * np.cos(np.arange(box[0]) * 0.37)[None, None, :] * np.ones((box[2], box[1], 1))
    return rho * (1.0 + 0.05 * rng.uniform(-1, 1, size=rho.shape))


@pytest.mark.parametrize("box,prec,rows", [
    ((256, 3, 1400), "f32", 3), ((335, 3, 2000), "f32", 2), ((335, 5, 1200), "f32", 3), ((257, 10, 700), "f32", 4),
    ((564, 48, 48), "f32", 1), ((549, 100, 100), "f32", 1), ((107, 108, 109), "f32", 12),
    ((3, 640, 641), "f32", 320), ((80, 80, 80), "f32", 16), ((100, 93, 87), "f32", None),
    ((256, 4, 300), "f16", 4), ((512, 3, 300), "f16", 2), ((640, 48, 48), "f16", 1), ((56, 66, 60), "f16", 14),
])
def test_planned_boxes(box, prec, rows):
    plan = launch_rules.row_plan(prec, box)
    assert plan and (rows is None or plan["by"] == rows)
    assert launch_rules.step_route(prec, box) == 1
    fields, rho = [], field(box)
    for fixed in (False, True):
        lat = P.Lattice(*box, G=-5.0, prec=prec)
        try:
            if fixed:
                code = lat.get_tile()
                lat.set_tile(code + 10 * min(8, box[2]) if code // 10 ** 8 == 5 or box[0] >= 32 else 132080001)
            lat.init_rho(rho)
            lat.step(5)
            fields.append(lat.get_populations())
            assert not (lat.observables().status_bits & 16)
        finally:
            lat.close()
    assert np.isfinite(fields[0]).all() and np.array_equal(*fields)


@pytest.mark.parametrize("boxes,mode", [
    ([(64, 64, 64), (72, 40, 33), (96, 24, 50)], ROW),
    ([(65, 65, 65), (61, 70, 66), (97, 50, 61), (64, 64, 64)], ROW_ANY),
])
def test_groups(boxes, mode):
    assert launch_rules.batch_mix("f32", 4, boxes)[0] == mode
    lats = [[P.Lattice(*b, G=-5.0, prec="f32") for b in boxes] for _ in range(2)]
    try:
        for both in zip(*lats):
            for lat in both:
                lat.init_drop([lat.nx // 2, lat.ny // 2, lat.nz // 2], 8.0, 1.85, 0.13)
        g = P.Group(lats[0])
        for n in (1, 6, 130):
            g.step(n)
            for lat in lats[1]:
                lat.step(n)
        for a, b in zip(*lats):
            pa = a.get_populations()
            assert np.isfinite(pa).all() and np.array_equal(pa, b.get_populations())
        g.close()
    finally:
        for lat in lats[0] + lats[1]:
            lat.close()
