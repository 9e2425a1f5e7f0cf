"""Scattering where the densities are small: well channeled particles stay far from the planes or strings, and all of
their v_y (their whole transverse motion across the plane's field) comes from kicks that follow the
densities' tails. Against the trajectory oracle; tolerance 1e-9 of a field's scale per particle, as for the other
FP64 records, with the oracle's own exponentials good to some units in the last place of their arguments (up to 170: 4e-14)."""
import numpy as np
import pytest

from oracle import traj as T
import paper_1910_10391_gb300 as rad
from paper_1910_10391_gb300 import inputs as I

from test_crystal_gpu import D_P, MS, channel, potentials, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [24, 2433])
def test_planar_kicks_between_the_planes(n):
    """Positrons entering parallel to the planes at 2 to 12.8 thermal amplitudes from the nearest one; eight lanes
    and one lane per particle."""
    E, dt, L = 10e9, 5e-9, 60
    lib, orc = potentials()
    x0 = np.resize(np.linspace(2 * I.RHO_THERMAL, D_P / 2, 24), n)
    got, _, off = run_gpu(channel(+1, MS), lib, x0, np.zeros(n), E, np.full(n, L), dt, 5)
    for p in list(range(24)) + [n - 1]:
        ref = T.trajectories(x0[p:p + 1], np.zeros(1), 0.0, E, L, dt, 5, charge=+1, ms=True, pot=orc,
                             particle_ids=np.array([p], dtype=np.int64))[0]
        g = got[off[p]:off[p + 1]]
        for f in ("y", "vy", "ay"):
            i = I.FIELDS.index(f)
            scale = np.abs(ref[:, i]).max()
            assert scale > 0.0
            assert np.abs(g[:, i] - ref[:, i]).max() <= 1e-9 * scale, (p, f, x0[p] / I.RHO_THERMAL)
