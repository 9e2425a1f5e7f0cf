"""Planar trajectories whose fit the table of the potential does not resolve (tab_fits in rad_traj.cu) and fits next to its
two bounds, below 4096 particles (a group of eight lanes each in the direct form) and from there on (one lane),
against the trajectory oracle. Bounds: h^2 k <= 0.0197 for the narrowest Gaussian e^{-k r^2}, h = d_p / 256, and
k d_p^2 <= 125 for the widest of the force. Tolerance 1e-9 of a field's scale per particle, as for the FP64
records elsewhere."""
import math

import numpy as np
import pytest

from oracle import traj as T
import paper_1910_10391_gb300 as rad
from paper_1910_10391_gb300 import inputs as I

from test_crystal_gpu import ALL, D_P, EL, LL, LOSS, MS, entries, run_gpu

pytestmark = pytest.mark.gpu


def check(got, off, picks, x0, th, E, L, dt, seed, charge, flags, orc, rho):
    for p in picks:
        ref = T.trajectories(x0[p:p + 1], th[p:p + 1], 0.0, E, L, dt, seed, charge=charge, rho=rho, ms=bool(flags & MS),
                             ll=bool(flags & LL), ms_loss=bool(flags & LOSS), ms_el=bool(flags & EL), pot=orc,
                             particle_ids=np.array([p], dtype=np.int64))[0]
        g = got[off[p]:off[p + 1]]
        err = np.abs(g - ref).max(0) / np.maximum(np.abs(ref).max(0), 1e-300)
        assert np.all(err <= 1e-9), (p, err)


@pytest.mark.parametrize("n,L", [(24, 300), (2433, 24), (4096, 12)])
@pytest.mark.parametrize("h2k", [0.0195, 0.0199, 0.05])
@pytest.mark.parametrize("charge", [+1, -1])
def test_narrow_terms(n, L, h2k, charge):
    """The fit's last terms have b = 0, so that 1 / rho^2 is its largest k; the first of the three fits in."""
    E, dt, seed = 20e9, 5e-9, 9
    rho = D_P / 256 / math.sqrt(h2k)
    b, bx = I.SYNTH_DT_B[:3] + (0.0,), I.SYNTH_DT_BX[:3] + (0.0,)
    lib = rad.RadPlanarPotential.make(I.SYNTH_DT_A, b, I.SI_N, I.SYNTH_DT_AX, bx, I.SYNTH_DT_CX, I.SI_I_EV, n_neighbours=3)
    orc = T.PlanarPotential(I.SYNTH_DT_A, b, I.SI_N, I.SYNTH_DT_AX, bx, I.SYNTH_DT_CX, I.SI_I_EV, K=3)
    x0, th = entries(n, E, 4)
    ch = rad.RadChannel(0.0, D_P, I.EPS_S_EV, I.SI_X0, rho, I.ME_EV, charge, ALL)
    got, _, off = run_gpu(ch, lib, x0, th, E, np.full(n, L), dt, seed)
    check(got, off, sorted({0, 1, n // 2, n - 2, n - 1}), x0, th, E, L, dt, seed, charge, ALL, orc, rho)


@pytest.mark.parametrize("n", [24, 4096])
@pytest.mark.parametrize("kd2", [120.0, 130.0, 600.0])
def test_no_wide_term(n, kd2):
    """One narrow Gaussian: the force between the planes is its tail, and particles that enter parallel to the planes
    follow it; the first of the three fits in."""
    E, dt, L = 20e9, 5e-9, 40
    C = D_P * D_P / kd2
    b = ((C - I.RHO_THERMAL ** 2) * 4 * math.pi ** 2,) if kd2 < 600 else (0.0,)
    rho = I.RHO_THERMAL if kd2 < 600 else math.sqrt(C)
    lib = rad.RadPlanarPotential.make((3e-10,), b, I.SI_N, n_neighbours=2)
    orc = T.PlanarPotential((3e-10,), b, I.SI_N, K=2)
    x0 = np.resize(np.linspace(0.05, 0.48, 24) * D_P, n)
    ch = rad.RadChannel(0.0, D_P, I.EPS_S_EV, I.SI_X0, rho, I.ME_EV, +1, 0)
    got, _, off = run_gpu(ch, lib, x0, np.zeros(n), E, np.full(n, L), dt, 1)
    check(got, off, range(24), x0, np.zeros(n), E, L, dt, 1, +1, 0, orc, rho)


def test_wide_term_without_weight():
    """A padded fit: the wide Gaussian has no amplitude, the narrow one's tail is the force between the planes."""
    E, dt, L, n = 20e9, 5e-9, 40, 24
    rho = D_P / math.sqrt(600.0)
    a, b = (3e-10, 0.0), (0.0, 4e-20)
    lib = rad.RadPlanarPotential.make(a, b, I.SI_N, n_neighbours=2)
    orc = T.PlanarPotential(a, b, I.SI_N, K=2)
    x0 = np.linspace(0.05, 0.48, n) * D_P
    ch = rad.RadChannel(0.0, D_P, I.EPS_S_EV, I.SI_X0, rho, I.ME_EV, +1, 0)
    got, _, off = run_gpu(ch, lib, x0, np.zeros(n), E, np.full(n, L), dt, 1)
    check(got, off, range(n), x0, np.zeros(n), E, L, dt, 1, +1, 0, orc, rho)
