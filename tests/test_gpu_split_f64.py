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


@pytest.mark.parametrize("box,stencil,prec", [
    ((21, 13, 11), "E4", "f64"), ((24, 20, 16), "E4", "f32"), ((23, 20, 16), "E6", "f32"), ((20, 16, 12), "E8", "f64"),
])
def test_a_workspace_without_the_psi_plane_still_steps(box, stencil, prec):
    """lbm_create takes a workspace that ends before the psi plane (and nothing
    shorter); its steps run the tile kernels, bitwise the same."""
    import torch
    from paper_2105_08772_gb300 import _lib, lbm
    f0 = inputs.random_populations(box[::-1], seed=sum(box))
    rho = f0.sum(axis=0)
    st, pr = _lib.STENCILS[stencil], _lib.PRECS[prec]
    cbox, eos = lbm.make_box(*box), lbm.make_eos("one_minus_exp")
    full = lbm.lbm_workspace_bytes(cbox, st, pr)
    plane = box[0] * box[1] * box[2] * (8 if prec == "f64" else 4)
    short = full - (plane + (-plane) % 256)
    ws = torch.empty(full + 256, dtype=torch.uint8, device="cuda")
    ptr = ws.data_ptr() + (-ws.data_ptr()) % 256
    stream = torch.cuda.current_stream().cuda_stream
    with pytest.raises(P.LBMError):
        lbm.lbm_create(cbox, 1.0, -5.0, eos, st, pr, ptr, short - 1, stream)
    fields = []
    for nbytes in (full, short):
        ctx = lbm.lbm_create(cbox, 1.0, -5.0, eos, st, pr, ptr, nbytes, stream)
        try:
            lbm.lbm_init_rho(ctx, rho)
            lbm.lbm_step(ctx, 7)
            fields.append(lbm.lbm_get_populations(ctx, np.empty((19,) + box[::-1])))
        finally:
            lbm.lbm_destroy(ctx)
    assert np.isfinite(fields[0]).all() and np.array_equal(*fields)
