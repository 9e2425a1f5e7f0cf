"""The kernels that sum over runs of samples (rad_cheb.cu, rad_mixed_nodes.cu) against the direct kernels of the same
form in how far they are from the exact sum: the reference reduces every phase in extended precision
(numpy.longdouble), which the FP64 oracle, whose rounded phases the direct kernels share, does not.

"top" has all energies next to the highest one of their tile, which sees the most of a dropped term.

Bound: the 2-norm of the cube's error and the median error of a bin (floor 1e-6 of the peak) are at most 1.1 times the
direct kernel's, a tenth for the scatter of a rounding error over some thousand bins, or 4.4e-16, two units in
the last place of an FP64 result."""
import functools

import numpy as np
import pytest

import paper_1910_10391_gb300 as rad
from paper_1910_10391_gb300 import inputs as I

from test_cut_gpu import cube_of, plan_of

pytestmark = pytest.mark.gpu
LD = np.longdouble
TWO_PI = LD("6.283185307179586476925286766559005768394")


def directions(n):
    g = I._ensemble_grid(10e9, 20.0, 8, 12)
    pick = np.linspace(0, g.theta_x.size - 1, n).astype(int)
    return g.theta_x[pick].copy(), g.theta_y[pick].copy(), g.d_omega[pick].copy()


@functools.lru_cache(maxsize=None)
def case(kind, mode):
    if kind == "undulator":
        tr = I.weak_undulator(1000.0, 0.5e-10, 10e-6, 5, 4096)
        grid = I.make_grid(I.omega_linear(96, 1.2 * I.undulator_first_harmonic_eV(1000.0, 0.5e-10, 10e-6)), 4, 4, 2e-3)
    else:
        tr = I.channeling(2, 10e9, +1, 3000, 5e-9, 3)
        hw = {"positrons": I.omega_log(96, 1e6, 1e9), "top": np.linspace(0.95e8, 1e8, 96),
              "narrow": np.linspace(4e9, 4.004e9, 96)}[kind]
        grid = I.Grid(hw, *directions(16))
    return tr, grid, exact_cube(tr, grid, mode)


def exact_cube(tr, grid, mode):
    hw, cube = np.asarray(grid.hbar_omega_eV, LD), 0.0
    for p in range(tr.n_particles):
        t, x, y, dz, vx, vy, dvz, ax, ay, az = np.asarray(tr.samples[tr.offsets[p]:tr.offsets[p + 1]], LD).T
        g, E = LD(tr.gamma[p]), LD(tr.energy_eV[p])
        w = np.concatenate([t[1:2] - t[:1], t[2:] - t[:-2], t[-1:] - t[-2:-1]]) / 2
        u = hw / E
        ws = hw / LD(1.973269804e-7) / (1 if mode == rad.RAD_CLASSICAL else 1 - u)
        S = np.empty((hw.size, grid.theta_x.size))
        for j, (nx, ny) in enumerate(zip(np.asarray(grid.theta_x, LD), np.asarray(grid.theta_y, LD))):
            c = 1 / (2 * g * g) + (nx * nx + ny * ny) / 2
            A = c * t - dz - nx * x - ny * y
            D = c - dvz - nx * vx - ny * vy
            m = az + nx * ax + ny * ay
            fx, fy = ((nx - vx) * m - ax * D) / (D * D) * w, ((ny - vy) * m - ay * D) / (D * D) * w
            f = np.stack([fx, fy, -(nx * fx + ny * fy), m / (D * D) * w], 1).astype(np.float64)
            ph = ws[:, None] * A
            ph = (ph - np.rint(ph / TWO_PI) * TWO_PI).astype(np.float64)
            q = (np.cos(ph) @ f) ** 2 + (np.sin(ph) @ f) ** 2
            I2 = q[:, :3].sum(1)
            if mode != rad.RAD_CLASSICAL:
                v = u.astype(np.float64)
                I2 = 0.5 * (1 + (1 - v) ** 2) * I2 + v * v / (2 * float(g) ** 2) * q[:, 3]
            S[:, j] = I2
        cube = cube + float(tr.weight[p]) * S
    return cube * (7.2973525693e-3 / (4 * np.pi ** 2))


def errors(got, ref):
    e = np.abs(got - ref)
    return np.linalg.norm(e) / np.linalg.norm(ref), np.median(e / np.maximum(ref, 1e-6 * ref.max()))


@pytest.mark.parametrize("form", [rad.RAD_FP64, rad.RAD_FP64_DF, rad.RAD_MIXED])
@pytest.mark.parametrize("kind,mode", [("undulator", rad.RAD_CLASSICAL), ("positrons", rad.RAD_CLASSICAL),
                                       ("positrons", rad.RAD_SPIN_HALF), ("top", rad.RAD_CLASSICAL),
                                       ("top", rad.RAD_SPIN_HALF)])
def test_no_further_from_the_exact_sum_than_directly(form, kind, mode):
    tr, grid, ref = case(kind, mode)
    inp = rad.DeviceInputs(tr, grid)
    p, _ = plan_of(inp, mode, form)
    err = {}
    for cut in (0, inp.n_omega):
        assert p.set_cut(cut) == rad.RAD_OK
        err[cut] = errors(cube_of(p, inp), ref)
        assert p.last_cut() == cut
    p.close()
    print(err)
    assert all(r <= max(1.1 * d, 4.4e-16) for r, d in zip(err[inp.n_omega], err[0])), err


@pytest.mark.parametrize("form", [rad.RAD_FP64, rad.RAD_FP64_DF, rad.RAD_MIXED])
def test_long_trajectory_in_one_piece(form):
    """Per-particle spectra keep a trajectory in one piece, so that its amplitudes collect some hundred runs."""
    import torch
    tr = I.channeling(2, 10e9, +1, 12000, 5e-9, 3)
    grid = I.Grid(I.omega_log(96 if form == rad.RAD_MIXED else 64, 1e7, 1e9), *directions(16))
    ref = exact_cube(tr, grid, rad.RAD_SPIN_HALF)
    inp = rad.DeviceInputs(tr, grid)
    p, _ = plan_of(inp, rad.RAD_SPIN_HALF, form, rad.RAD_PER_PARTICLE | 2)
    err = {}
    for cut in (0, inp.n_omega):
        assert p.set_cut(cut) == rad.RAD_OK
        out = torch.full((2, inp.n_omega), np.nan, dtype=torch.float64, device="cuda")
        assert p.execute(*inp.args(), None, out, None, None) == rad.RAD_OK
        assert p.last_cut() == cut
        err[cut] = errors(out.cpu().numpy().sum(0), ref @ grid.d_omega)
    p.close()
    print(err)
    assert all(r <= max(1.1 * d, 4.4e-16) for r, d in zip(err[inp.n_omega], err[0])), err


@pytest.mark.parametrize("mode", [rad.RAD_CLASSICAL, rad.RAD_SPIN_HALF])
def test_nodes_of_a_narrow_band(mode):
    """A band far above its width: the node form's phases about a run's centre reach (centre / spacing) pi / 2, up to the
    whole range that the direct form sees from its window's reference, and its error stays below that form's."""
    test_no_further_from_the_exact_sum_than_directly(rad.RAD_MIXED, "narrow", mode)
