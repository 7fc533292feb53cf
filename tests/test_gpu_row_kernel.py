"""The whole-row step kernel (lbm_kernels_row.cuh) against the moment kernel.

Tile kinds 5 and 6 with a launcher-chosen z chunk take the row kernel on boxes
that it has a cut for; a fixed z chunk of the same kinds takes the moment kernel.
Both do the same operations per node, so the fields are bitwise equal -- on
aligned and unaligned rows, with one or several rows per item, blocks that wrap in
y, rows of 3 or 4 nodes, few planes, several rounds of items, and after odd and
even step counts (the row kernel walks every other step downwards).
"""
import numpy as np
import pytest

import paper_2105_08772_gb300 as P

pytestmark = pytest.mark.gpu


# boxes that take the two passes (lbm_kernels_split.cuh) where the others take the row
# kernel, with their stencil and tau: for tau != 1 a fixed z chunk runs the chunked
# (aligned rows) or the pipelined kernel
OTHER = {
    (72, 60, 64): ("E4", 0.8), (71, 60, 64): ("E4", 1.3), (3, 250, 261): ("E4", 0.7), (335, 41, 23): ("E4", 0.8),
    (68, 60, 64): ("E6", 1.0), (69, 60, 64): ("E6", 1.0), (256, 31, 25): ("E6", 1.0), (8, 170, 150): ("E6", 1.0),
    (3, 3, 3): ("E4", 1.0), (37, 29, 23): ("E4", 1.0), (100, 3, 4): ("E4", 1.0), (57, 57, 58): ("E4", 1.0),
    (68, 64, 60): ("E8", 1.0), (61, 64, 60): ("E8", 1.0), (5, 201, 199): ("E8", 1.0), (68, 60, 63): ("E6", 0.8),
}


@pytest.mark.parametrize("box,prec,zc", [(b, "f32", min(8, b[2])) for b in OTHER] + [
    ((64, 56, 56), "f32", 8),        # aligned, 16 rows an item
    ((61, 60, 60), "f32", 8),        # unaligned rows
    ((127, 41, 43), "f32", 7),       # unaligned, ragged last row block and chunk
    ((4, 240, 240), "f32", 0),       # rows of 4 (kind 6 default; its twin: kind 1)
    ((3, 260, 260), "f32", 0),       # rows of 3
    ((200, 3, 400), "f32", 16),      # three rows: a block wraps on both sides
    ((201, 3, 400), "f32", 16),
    ((256, 256, 3), "f32", 3),       # three planes
    ((440, 24, 24), "f32", 8),       # long rows: two an item
    ((335, 41, 24), "f32", 8),
    ((600, 20, 20), "f32", 8),       # longer than a row item
    ((76, 72, 70), "f32", 8),        # boxes from here on are large enough for rows in F32
    ((107, 108, 109), "f32", 8),     # (above: the two passes)
    ((127, 99, 97), "f32", 7),
    ((4, 300, 300), "f32", 0),
    ((3, 640, 641), "f32", 0),
    ((200, 3, 600), "f32", 16),
    ((201, 3, 2000), "f32", 16),
    ((256, 456, 3), "f32", 3),
    ((440, 30, 28), "f32", 8),
    ((335, 41, 90), "f32", 8),
    ((600, 51, 50), "f32", 8),       # too long, and too large for the two passes
    ((64, 64, 64), "f16", 8),
    ((56, 66, 60), "f16", 16),
    ((256, 40, 33), "f16", 16),
])
def test_row_kernel_is_bitwise_the_moment_kernel(box, prec, zc):
    rng = np.random.default_rng(sum(box))
    rho = 1.0 + 0.6 * np.cos(np.arange(box[0]) * 0.37)[None, None, :] * np.ones((box[2], box[1], 1))
    rho = rho * (1.0 + 0.05 * rng.uniform(-1, 1, size=rho.shape))
    fields = []
    for fixed in (False, True):
        stencil, tau = OTHER.get(box, ("E4", 1.0))
        lat = P.Lattice(*box, G=-5.0, prec=prec, stencil=stencil, tau=tau)
        try:
            code = lat.get_tile()
            assert code // 10 ** 8 in (5, 6) and code // 10 % 1000 == 0, code
            if fixed:
                lat.set_tile(code + 10 * zc if zc else 132080001)
            lat.init_rho(rho)
            lat.step(1)
            one = lat.get_populations()
            lat.step(8)
            fields.append((one, lat.get_populations()))
            assert not (lat.observables().status_bits & 16)
        finally:
            lat.close()
    for a, b in zip(*fields):
        assert np.isfinite(a).all() and np.array_equal(a, b)
