"""Frequency-node summation of the mixed form (rad_mixed_nodes.cu) against the oracle, where its
tiling can go wrong: 128-energy tiles one short of, at and one past their end, windows of 256 samples
the same, particles of two samples, narrow bands far above their width, equal energies, and descending energies (which take the direct form).

Tolerance: the mixed form's contract (assert_mixed_close, 1e-4 of a bin). The node form's own part of
it is the interpolation's truncation, 2.6e-7 of |f| per sample, and FP32 phases below 90 rad
(5e-6 rad)."""
import numpy as np
import pytest

import oracle as O
import paper_1910_10391_gb300 as rad
from paper_1910_10391_gb300 import inputs as I

from helpers import MODE_ORC, assert_mixed_close, gpu_cube

pytestmark = pytest.mark.gpu


def bunch(lens, seed=5):
    src = I.channeling(len(lens), 10e9, +1, 3000, 5e-9, seed=seed)
    parts = [I.single(np.ascontiguousarray(src.samples[src.offsets[p]:src.offsets[p] + n]), src.gamma[p])
             for p, n in enumerate(lens)]
    tr = I.concat(parts)
    tr.energy_eV = src.energy_eV.copy()
    return tr


@pytest.mark.parametrize("mode", [rad.RAD_CLASSICAL, rad.RAD_SPIN0, rad.RAD_SPIN_HALF])
@pytest.mark.parametrize("n_omega", [96, 127, 128, 129, 256, 257, 513])
def test_energy_tiles(mode, n_omega):
    tr = bunch([255, 256, 257, 700])
    grid = I._ensemble_grid(10e9, 20.0, n_omega, 5)
    got = gpu_cube(tr, grid, mode, rad.RAD_MIXED)["cube"]
    assert_mixed_close(got, O.spectrum_cube(tr, grid, MODE_ORC[mode]))


@pytest.mark.parametrize("mode", [rad.RAD_CLASSICAL, rad.RAD_SPIN_HALF])
@pytest.mark.parametrize("lens", [[2, 3, 31, 33, 65], [2999]])
def test_runs(mode, lens):
    tr = bunch(lens)
    grid = I._ensemble_grid(10e9, 20.0, 160, 4)
    got = gpu_cube(tr, grid, mode, rad.RAD_MIXED)["cube"]
    assert_mixed_close(got, O.spectrum_cube(tr, grid, MODE_ORC[mode]))


@pytest.mark.parametrize("kind", ["narrow", "equal", "descending", "linear"])
def test_energy_grids(kind):
    tr = bunch([520, 300])
    hw = {"narrow": 1e8 * np.linspace(1.0, 1.001, 130), "equal": np.full(130, 2e8),
          "descending": I.omega_log(130, 1e6, 5e9)[::-1], "linear": I.omega_linear(130, 2e9)}[kind]
    g = I._ensemble_grid(10e9, 20.0, 8, 4)
    grid = I.Grid(np.ascontiguousarray(hw), g.theta_x, g.theta_y, g.d_omega)
    got = gpu_cube(tr, grid, rad.RAD_SPIN_HALF, rad.RAD_MIXED)["cube"]
    assert_mixed_close(got, O.spectrum_cube(tr, grid, O.SPIN_HALF))
