"""Which kernels a batch may run: no mode is offered for a box that its kernel does
not take.  The row-chunk moment kernel (mode 2) stages a tile's rows in 16-byte
chunks that wrap in x at most once, so it needs nx % 4 == 0 and nx >= 40 (FP16:
nx % 8 == 0 and nx >= 48), whatever kernel the set would get by default."""
import itertools

import pytest

import launch_rules

MIXED, UNIT, MOMENT, ELEM, ROW, ROW_ANY = range(6)


@pytest.mark.parametrize("boxes,mode,tuned", [
    ([(32, 32, 32)] * 6, ROW, {ROW, ELEM, UNIT}),
    ([(16, 64, 64)] * 4, ROW, {ROW, ELEM, UNIT}),
    ([(64, 64, 64), (32, 32, 32)], ROW, {ROW, ELEM, UNIT}),
    ([(64, 64, 64), (40, 32, 32)], ROW, {ROW, MOMENT, ELEM, UNIT}),
    ([(64, 64, 64), (33, 32, 32)], ROW_ANY, {ROW_ANY, ELEM, UNIT}),
    ([(48, 40, 36), (40, 32, 28)], MOMENT, {MOMENT, ELEM, UNIT}),
    ([(32, 32, 32)] * 5, ELEM, {ELEM, UNIT}),
])
def test_f32_sets(boxes, mode, tuned):
    assert launch_rules.batch_mix("f32", 4, boxes, slots=2)[::2] == (mode, tuned)


def test_f16_f64_and_mixed_tau_sets():
    assert launch_rules.batch_mix("f16", 4, [(64, 64, 64)], slots=1)[::2] == (ROW, {ROW, MOMENT})
    assert launch_rules.batch_mix("f16", 4, [(64, 40, 36)], slots=1)[::2] == (MOMENT, {MOMENT})
    assert launch_rules.batch_mix("f64", 4, [(64, 64, 64)])[::2] == (MOMENT, {MOMENT, ELEM, UNIT})
    assert launch_rules.batch_mix("f64", 6, [(37, 64, 64)])[::2] == (ELEM, {ELEM, UNIT})
    assert launch_rules.batch_mix("f32", 4, [(64, 64, 64)] * 2, [1.0, 0.8])[::2] == (MIXED, {MIXED})


@pytest.mark.parametrize("prec,stencil", [("f32", 4), ("f32", 6), ("f32", 8), ("f64", 4), ("f64", 8)])
def test_every_offered_mode_takes_every_box(prec, stencil):
    """All pairs of a small and a large box: offered modes are modes that take both, and
    the row-chunk moment kernel is never among them for a row it cannot stage."""
    m = 3 if stencil == 4 else 5
    small = [(m, m, m), (8, 9, 10), (16, 16, 16), (36, 12, 12), (38, 8, 8), (40, 8, 8), (41, 8, 8), (600, 8, 8)]
    large = [(16, 128, 128), (32, 96, 96), (33, 96, 96), (64, 64, 64), (61, 64, 64), (600, 30, 30)]
    for a, b in itertools.product(small, large):
        mode, takes, cand = launch_rules.batch_mix(prec, stencil, [a, b])
        assert mode in cand and cand <= takes
        chunks = all(box[0] % 4 == 0 and box[0] >= 40 for box in (a, b))
        assert (MOMENT in takes) == chunks
        rows = prec == "f32" and stencil == 4 and all(box[0] < 600 for box in (a, b))
        assert (ROW_ANY in takes) == rows
        assert (ROW in takes) == (rows and all(box[0] % 4 == 0 for box in (a, b)))


@pytest.mark.parametrize("boxes,slots,rows", [
    # groups
    ([(8, 8, 8)] * 391, 0, False), ([(16, 16, 16)] * 48, 0, False), ([(20, 20, 20)] * 100, 0, False),
    ([(24, 24, 24)] * 14, 0, False), ([(32, 32, 32)] * 6, 0, False), ([(64, 3, 64)] * 100, 0, False),
    ([(461, 48, 48)] * 4, 0, False), ([(65, 65, 65)], 0, False), ([(64, 64, 64), (65, 65, 65)], 0, False),
    ([(33, 33, 33)] * 8, 0, True), ([(40, 40, 40)] * 5, 0, True), ([(32, 32, 32)] * 60, 0, True),
    ([(64, 64, 64)] * 4, 0, True), ([(65, 65, 65)] * 3, 0, True), ([(128, 128, 128)] * 2, 0, True),
    ([(s, s, s) for s in (64, 72, 80, 96, 112, 128)], 0, True),
    # batches: the tile kernels' z chunks of 16 planes leave few small items
    ([(16, 16, 16)] * 48, 8, True), ([(16, 16, 16)] * 48, 48, False), ([(8, 8, 8)] * 400, 100, False),
    ([(24, 24, 24)] * 64, 2, True), ([(24, 24, 24)] * 60, 60, True), ([(64, 3, 64)] * 20, 20, False),
    ([(64, 64, 64)] * 4, 1, True), ([(97, 97, 97)] * 4, 4, True),
])
def test_the_row_kernel_gets_the_sets_it_is_faster_on(boxes, slots, rows):
    """Measured on both sides of the line (GB300)."""
    assert (launch_rules.batch_mix("f32", 4, boxes, slots=slots)[0] in (ROW, ROW_ANY)) == rows
