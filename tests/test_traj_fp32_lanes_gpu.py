"""The FP32 form of planar trajectories on one lane per particle (k_channel_mixed<true, 1>: from 2433 particles on, or
with more than four neighbouring planes), which its tests of some dozen particles do not reach. Both forms add the
same terms in the same order, so the first particles of a large ensemble have the records of the same
particles alone, bit for bit; the form with five neighbours is compared with the oracle under the FP32 form's
tolerances."""
import numpy as np
import pytest

import paper_1910_10391_gb300 as rad
from paper_1910_10391_gb300 import inputs as I

from test_crystal_gpu import ALL, FP32, MIXED_TOL_MS, channel, entries, field_errors, oracle, potentials, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("terms,K", [(4, 3), (3, 3), (4, 1), (4, 4), (1, 2)])
@pytest.mark.parametrize("charge", [+1, -1])
def test_one_lane_equals_eight(terms, K, charge):
    E, dt, L, n = 20e9, 5e-9, 60, 2433
    lib = rad.RadPlanarPotential.make(I.SYNTH_DT_A[:terms], I.SYNTH_DT_B[:terms], I.SI_N, I.SYNTH_DT_AX[:terms],
                                      I.SYNTH_DT_BX[:terms], I.SYNTH_DT_CX, I.SI_I_EV, n_neighbours=K)
    x0, th = entries(n, E, 12)
    out = [run_gpu(channel(charge, ALL | FP32), lib, x0[:m], th[:m], E, np.full(m, L), dt, 3) for m in (24, 2432, n)]
    for rec, energy, _ in out[:2]:
        assert np.array_equal(rec, out[2][0][:rec.shape[0]])
        assert np.array_equal(energy, out[2][1][:energy.shape[0]])


def test_five_neighbours():
    n, dt, E, seed, L = 24, 5e-9, 20e9, 21, 3000
    lib, orc = potentials(K=5)
    x0, th = entries(n, E, 8)
    got, _, _ = run_gpu(channel(+1, ALL | FP32), lib, x0, th, E, np.full(n, L), dt, seed)
    ref, _ = oracle(orc, x0, th, E, L, dt, seed, +1, ALL)
    worst = field_errors(got.reshape(n, L, 10), ref)
    for name, t in MIXED_TOL_MS.items():
        assert worst[name] <= t, (name, worst[name])
