"""Chebyshev-moment summation of the FP64 forms (rad_cheb.cu) against the oracle where its tiling can go
wrong: direction tiles of 32 one short of, at and one past their end, energy tiles (256 or 512) the
same, windows of 256 samples the same, particles of two samples (runs shorter than the four warps of
a block), several particles with their own energies, a grid the direct kernel shares, and descending
energies (which take the direct form).

Tolerance: the FP64 forms' contract, 1e-9 of a bin with a floor of 1e-6 of the peak. The series'
first dropped term is below 1e-14 of |f|."""
import numpy as np
import pytest

import oracle as O
import paper_1910_10391_gb300 as rad
from paper_1910_10391_gb300 import inputs as I

from helpers import MODE_ORC, assert_fp64_close, gpu_cube

pytestmark = pytest.mark.gpu
FORMS = [rad.RAD_FP64, rad.RAD_FP64_DF]


def bunch(lens, seed=5):
    src = I.channeling(len(lens), 10e9, +1, 1100, 5e-9, seed=seed)
    tr = I.concat([I.single(np.ascontiguousarray(src.samples[src.offsets[p]:src.offsets[p] + n]), src.gamma[p])
                   for p, n in enumerate(lens)])
    tr.energy_eV = src.energy_eV * np.linspace(1.0, 0.9, len(lens))
    return tr


def directions(n, hw):
    g = I._ensemble_grid(10e9, 20.0, 8, 8)
    pick = np.arange(n) % g.theta_x.size
    return I.Grid(np.ascontiguousarray(hw), g.theta_x[pick].copy(), g.theta_y[pick].copy(), g.d_omega[pick].copy())


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("n_angles", [16, 31, 32, 33])
def test_direction_tiles(form, n_angles):
    tr = bunch([2, 3, 5, 255, 256, 257, 700])
    grid = directions(n_angles, I.omega_log(80, 1e5, 4e8))
    got = gpu_cube(tr, grid, rad.RAD_SPIN_HALF, form)["cube"]
    assert_fp64_close(got, O.spectrum_cube(tr, grid, O.SPIN_HALF))


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("mode,n_omega", [(rad.RAD_CLASSICAL, 512), (rad.RAD_CLASSICAL, 513), (rad.RAD_SPIN0, 65),
                                          (rad.RAD_SPIN_HALF, 256), (rad.RAD_SPIN_HALF, 257)])
def test_energy_tiles(form, mode, n_omega):
    tr = bunch([300, 40])
    grid = directions(16, I.omega_log(n_omega, 1e5, 5e8))
    got = gpu_cube(tr, grid, mode, form)["cube"]
    assert_fp64_close(got, O.spectrum_cube(tr, grid, MODE_ORC[mode]))


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("kind", ["linear", "wide", "equal", "descending"])
def test_energy_grids(form, kind):
    """One particle in time pieces; 'wide' reaches energies that the direct kernel sums."""
    tr = bunch([1031])
    hw = {"linear": I.omega_linear(130, 2e8), "wide": I.omega_log(300, 1e6, 5e9), "equal": np.full(130, 2e8),
          "descending": I.omega_log(130, 1e6, 5e9)[::-1]}[kind]
    grid = directions(40, hw)
    got = gpu_cube(tr, grid, rad.RAD_SPIN_HALF, form)["cube"]
    assert_fp64_close(got, O.spectrum_cube(tr, grid, O.SPIN_HALF))
