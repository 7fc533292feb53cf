"""lbm_batch_run on queues that the row kernel takes, with fewer slots than runs (slots
are refilled while others run), plain and tuned: every lattice ends bitwise as it does
alone.  After tuning the batch runs one of the modes that take every box of the queue,
so queues with rows too short for the row-chunk moment kernel are among them."""
import pytest

import launch_rules
import paper_2105_08772_gb300 as P

pytestmark = pytest.mark.gpu

KEYS = ("n_in", "n_out", "P_in", "P_out", "dP", "mass", "R_e", "C", "D", "max_u")
ROW, ROW_ANY = 4, 5
QUEUES = [   # storage, slots, boxes, kernel mode
    ("f32", 6, [(32, 32, 32)] * 4 + [(16, 64, 64)] * 3, ROW),
    ("f32", 3, [(64, 64, 64), (48, 40, 36), (72, 56, 31), (96, 24, 50), (40, 64, 64)], ROW),
    ("f32", 2, [(61, 60, 43), (33, 47, 29), (64, 64, 40), (85, 31, 50)], ROW_ANY),
    ("f16", 2, [(64, 64, 64), (48, 40, 36), (56, 66, 30), (128, 20, 41)], ROW),
    ("f16", 3, [(64, 16, 48)] * 4 + [(256, 9, 11)], ROW),
]


@pytest.mark.parametrize("tuned", [False, True])
@pytest.mark.parametrize("prec,slots,boxes,mode", QUEUES)
def test_batch_on_the_row_kernel_equals_single_runs(prec, slots, boxes, mode, tuned):
    assert launch_rules.batch_mix(prec, 4, boxes, slots=slots)[0] == mode
    runs = [(b, -5.0 - 0.1 * (k % 3), max(3.0, min(b) / 4.0), 1.9 - 0.05 * k) for k, b in enumerate(boxes)]
    batch = P.Batch(slots, tuple(max(b[a] for b in boxes) for a in range(3)), prec=prec)
    try:
        ids = [batch.enqueue(b, G=G, R=R, rho_in=ri, rho_out=0.13) for b, G, R, ri in runs]
        if tuned:   # the code names the kernel, of those that take every box
            code = batch.autotune(reps=2)
            offered = launch_rules.batch_mix(prec, 4, boxes, slots=slots)[2]
            assert mode in offered and code // 10 ** 6 in offered
            assert code // 1000 % 1000 in ((0, 8, 16, 32) if code // 10 ** 6 >= ROW else (8, 16, 32))
        batch.run(max_steps=96, check_every=48, tol_dP_rel=-1.0, tol_du=-1.0)
        for rid, (b, G, R, ri) in zip(ids, runs):
            status, got = batch.result(rid)
            assert status == P._lib.LBM_ENOTCONV and got.steps == 96 and not (got.status_bits & 16)
            lat = P.Lattice(*b, G=G, prec=prec)
            lat.init_drop([n // 2 for n in b], R, ri, 0.13)
            lat.step(96)
            want = lat.observables()
            assert all(getattr(got, k) == getattr(want, k) for k in KEYS), rid
            lat.close()
    finally:
        batch.close()
