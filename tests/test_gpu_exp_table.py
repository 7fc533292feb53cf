"""FP64 psi by table and series (lbm_exptab.cuh) at the edges of its range.

Densities on both sides of the table's limits (2^-6 and 7.9921875, for
psi = exp(-1/n) as 1/n), at table points and half-way between them, one step
against the oracle.  The densities reach 9 and the velocities order 1, so a
population is at most about 10; 64 roundings of that size are 7e-14, the bound.
"""
import numpy as np
import pytest

import paper_2105_08772_gb300 as P
from oracle import eos as E
from oracle import lbm3d

pytestmark = pytest.mark.gpu


def edge_values():
    x = [2.0 ** -6, 7.9921875, 1.0 / 64, 3.0 / 128, 5.0 / 128, 1.0, 1.0 + 1.0 / 128, 511.0 / 64, 9.0, 2.0 ** -7]
    x = np.array(x)
    return np.concatenate([x, np.nextafter(x, 0), np.nextafter(x, 10), x * (1 + 1e-9)])


@pytest.mark.parametrize("kind,G", [("one_minus_exp", -5.0), ("exp_inv", -9.2)])
def test_psi_table_edges_one_step(kind, G):
    shape = (6, 7, 9)
    v = edge_values()
    if kind == "exp_inv":
        v = 1.0 / v
        v = v[v < 20.0]          # 1/n at the table's edges; the densities stay below 20
    rng = np.random.default_rng(8)
    n = rng.choice(v, size=shape)
    if kind == "exp_inv":
        n = np.clip(n, 0.11, 20.0)
    f0 = lbm3d.init_from_density(n)
    lat = P.Lattice(shape[2], shape[1], shape[0], G=G, psi=kind)
    try:
        lat.set_populations(f0)
        lat.step(1)
        got = lat.get_populations()
    finally:
        lat.close()
    ref = lbm3d.step(f0, lbm3d.Model(tau=1.0, G=G, eos=E.EOS(kind)))
    scale = max(1.0, float(np.max(np.abs(ref))) / 10.0)
    assert np.max(np.abs(got - ref)) < 7e-14 * scale
