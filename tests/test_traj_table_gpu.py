"""Planar trajectories from the tabulated potential (k_channel_tab): particle counts around the block
grid and the switch from eight lanes to one lane per particle, positions far outside the first cell and
on cell borders and uneven lengths,
against the trajectory oracle. Tolerance as for the FP64 records elsewhere: 1e-9 of a field's scale
(the table's first dropped term is below 1e-16 of the narrowest Gaussian)."""
import numpy as np
import pytest

from oracle import traj as T
import paper_1910_10391_gb300 as rad
from paper_1910_10391_gb300 import inputs as I

from test_crystal_gpu import ALL, D_P, MS, channel, entries, potentials, run_gpu

pytestmark = pytest.mark.gpu


def check(got, off, picks, x0, th, lengths, E, dt, seed, charge, flags, orc):
    for p in picks:
        ref = T.trajectories(x0[p:p + 1], th[p:p + 1], 0.0, E, int(lengths[p]), dt, seed, charge=charge, ms=bool(flags & MS),
                             ll=bool(flags & rad.RAD_TRAJ_LL), ms_loss=bool(flags & rad.RAD_TRAJ_MS_LOSS),
                             ms_el=bool(flags & rad.RAD_TRAJ_MS_EL), pot=orc,
                             particle_ids=np.array([p], dtype=np.int64))[0]
        g = got[off[p]:off[p + 1]]
        scale = np.maximum(np.abs(ref).max(0), 1e-300)
        err = np.abs(g - ref).max(0) / scale
        assert np.all(err <= 1e-9), (p, err)


@pytest.mark.parametrize("n", [1, 151, 153, 2431, 2432])
def test_particle_counts(n):
    E, dt, seed = 10e9, 5e-9, 13
    lib, orc = potentials()
    x0, th = entries(n, E, 5)
    x0[0] = -1e4 * D_P + 0.3 * D_P
    if n > 3:
        x0[1], x0[2] = D_P, np.nextafter(D_P, 0.0)
    lengths = 30 + np.arange(n) % 7
    got, _, off = run_gpu(channel(+1, ALL), lib, x0, th, E, lengths, dt, seed)
    picks = sorted({0, min(1, n - 1), min(2, n - 1), n // 2, n - 1})
    check(got, off, picks, x0, th, lengths, E, dt, seed, +1, ALL, orc)


@pytest.mark.parametrize("K", [1, 8])
def test_neighbour_counts(K):
    E, dt = 20e9, 5e-9
    lib, orc = potentials(K=K)
    x0, th = entries(6, E, 8)
    lengths = np.full(6, 400)
    got, _, off = run_gpu(channel(-1, ALL), lib, x0, th, E, lengths, dt, 2)
    check(got, off, range(6), x0, th, lengths, E, dt, 2, -1, ALL, orc)


@pytest.mark.parametrize("n", [608, 609])
def test_axial_warp_and_half_warp(n):
    """Axial particles on both sides of the switch from a warp to 16 lanes each."""
    import test_axial_gpu as X
    lib, orc = X.potentials(K=1)
    E, dt = 10e9, 5e-9
    x0, y0, thx, thy = X.entries(n, E, orc.lat, seed=6)
    lengths = 20 + np.arange(n) % 5
    got, _, off = X.run_gpu(X.channel(-1, ALL), lib, x0, y0, thx, thy, E, lengths, dt, 4)
    for p in (0, 1, n // 2, n - 1):
        ref = T.axial_trajectories(x0[p:p + 1], y0[p:p + 1], thx[p:p + 1], thy[p:p + 1], E, int(lengths[p]), dt, 4, orc,
                                   charge=-1, ms=True, ms_el=True, ll=True, ms_loss=True,
                                   particle_ids=np.array([p], dtype=np.int64))
        X.close(got[off[p]:off[p + 1]], ref[0])
