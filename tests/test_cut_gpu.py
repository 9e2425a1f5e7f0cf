"""The moment kernel (rad_cheb.cu) and the frequency-node kernel (rad_mixed_nodes.cu) where their tiling can
go wrong, with the number of energies they sum set by rad_plan_set_cut and read back: direction tiles of 32 and
energy tiles (256 or 512; 128, 256 or 512) one short of, at and one past their end, windows of 256 samples the
same, particles of two samples, several particles with their own energies, narrow bands far above their
width, equal energies, energies too high for runs of more than one sample. Each case once with all energies and once
with a part of them, where one work item of the direct kernel is smaller than the grid.

Tolerances: the forms' contracts against the oracle, 1e-9 of a bin with a floor of 1e-6 of the peak (FP64 and
double-float) and 1e-4 of a bin (mixed)."""
import numpy as np
import pytest

import oracle as O
import paper_1910_10391_gb300 as rad
from paper_1910_10391_gb300 import inputs as I

from helpers import MODE_ORC, assert_fp64_close, assert_mixed_close
from test_cheb_gpu import bunch, directions
from test_nodes_gpu import bunch as bunch_nodes

pytestmark = pytest.mark.gpu
FORMS = [rad.RAD_FP64, rad.RAD_FP64_DF]
MODES = [rad.RAD_CLASSICAL, rad.RAD_SPIN0, rad.RAD_SPIN_HALF]


def plan_of(inp, mode, form, want=1, n_bins=0):
    p = rad.Plan(inp.n_samples, inp.n_particles, inp.n_omega, inp.n_angles, mode, form, want, n_bins)
    d = dict(kv.split("=") for kv in p.describe().split())
    return p, 32 * int(d["R"]) * (int(d["NW"]) if form == rad.RAD_FP64_DF else 1)


def cube_of(p, inp):
    import torch
    cube = torch.full((inp.n_omega, inp.n_angles), np.nan, dtype=torch.float64, device="cuda")
    assert p.execute(*inp.args(), cube, None, None, None) == rad.RAD_OK
    torch.cuda.synchronize()
    assert rad.rad_device_status(1) == rad.RAD_OK
    return cube.cpu().numpy()


def check(tr, grid, mode, form, ascending=True):
    ref = O.spectrum_cube(tr, grid, MODE_ORC[mode])
    inp = rad.DeviceInputs(tr, grid)
    p, gran = plan_of(inp, mode, form)
    n = inp.n_omega
    for cut in sorted({n, (n - 1) // gran * gran}):
        assert p.set_cut(cut) == rad.RAD_OK, cut
        assert f"cut={cut}" in p.describe().split()
        got = cube_of(p, inp)
        assert p.last_cut() == (cut if ascending else 0)
        (assert_mixed_close if form == rad.RAD_MIXED else assert_fp64_close)(got, ref)
    p.close()


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("n_angles", [16, 31, 32, 33])
@pytest.mark.parametrize("mode", [rad.RAD_CLASSICAL, rad.RAD_SPIN_HALF])
def test_moments_direction_tiles(form, n_angles, mode):
    tr = bunch([2, 3, 5, 255, 256, 257, 700])
    check(tr, directions(n_angles, I.omega_log(130, 1e5, 4e8)), mode, form)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("mode,n_omega", [(rad.RAD_CLASSICAL, 511), (rad.RAD_CLASSICAL, 512), (rad.RAD_CLASSICAL, 513),
                                          (rad.RAD_SPIN0, 65), (rad.RAD_SPIN0, 513), (rad.RAD_SPIN_HALF, 255),
                                          (rad.RAD_SPIN_HALF, 256), (rad.RAD_SPIN_HALF, 257)])
def test_moments_energy_tiles(form, mode, n_omega):
    check(bunch([300, 40]), directions(16, I.omega_log(n_omega, 1e5, 5e8)), mode, form)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("kind", ["linear", "wide", "narrow", "equal", "descending"])
def test_moments_energy_grids(form, mode, kind):
    """One particle in time pieces; 'wide' reaches energies whose runs are single samples."""
    hw = {"linear": I.omega_linear(130, 2e8), "wide": I.omega_log(300, 1e6, 5e9),
          "narrow": 1e8 * np.linspace(1.0, 1.001, 130), "equal": np.full(130, 2e8),
          "descending": I.omega_log(130, 1e6, 5e9)[::-1]}[kind]
    check(bunch([1031]), directions(40, hw), mode, form, ascending=kind != "descending")


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("n_omega", [96, 127, 128, 129, 255, 256, 257, 511, 512, 513])
def test_nodes_energy_tiles(mode, n_omega):
    check(bunch_nodes([255, 256, 257, 700]), I._ensemble_grid(10e9, 20.0, n_omega, 5), mode, rad.RAD_MIXED)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("lens", [[2, 3, 31, 33, 65], [63, 64, 65, 192, 193], [2999]])
def test_nodes_runs(mode, lens):
    check(bunch_nodes(lens), I._ensemble_grid(10e9, 20.0, 160, 4), mode, rad.RAD_MIXED)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("kind", ["narrow", "equal", "linear", "low", "descending"])
def test_nodes_energy_grids(mode, kind):
    hw = {"narrow": 1e8 * np.linspace(1.0, 1.001, 130), "equal": np.full(130, 2e8), "linear": I.omega_linear(130, 2e9),
          "low": I.omega_log(130, 1e3, 1e6), "descending": I.omega_log(130, 1e6, 5e9)[::-1]}[kind]
    g = I._ensemble_grid(10e9, 20.0, 8, 4)
    grid = I.Grid(np.ascontiguousarray(hw), g.theta_x, g.theta_y, g.d_omega)
    check(bunch_nodes([520, 300]), grid, mode, rad.RAD_MIXED, ascending=kind != "descending")


@pytest.mark.parametrize("form", FORMS + [rad.RAD_MIXED])
def test_per_particle(form):
    """Per-particle spectra: one chunk a particle, weights included."""
    import torch
    tr = bunch([300, 257, 2])
    tr.weight = np.array([1.0, 0.5, 2.0])
    grid = directions(33, I.omega_log(130, 1e5, 4e8))
    inp = rad.DeviceInputs(tr, grid)
    p, _ = plan_of(inp, rad.RAD_SPIN_HALF, form, rad.RAD_PER_PARTICLE | 2)
    assert p.set_cut(inp.n_omega) == rad.RAD_OK
    out = torch.full((3, inp.n_omega), np.nan, dtype=torch.float64, device="cuda")
    assert p.execute(*inp.args(), None, out, None, None) == rad.RAD_OK
    assert p.last_cut() == inp.n_omega
    assert rad.rad_device_status(1) == rad.RAD_OK
    ref = np.empty((3, inp.n_omega))
    for i in range(3):
        one = I.single(np.ascontiguousarray(tr.samples[tr.offsets[i]:tr.offsets[i + 1]]), tr.gamma[i])
        one.energy_eV, one.weight = tr.energy_eV[i:i + 1].copy(), tr.weight[i:i + 1].copy()
        ref[i] = O.spectrum_cube(one, grid, O.SPIN_HALF) @ grid.d_omega
    (assert_mixed_close if form == rad.RAD_MIXED else assert_fp64_close)(out.cpu().numpy(), ref)


@pytest.mark.parametrize("form", FORMS + [rad.RAD_MIXED])
def test_automatic_choice(form):
    """A call that fills the GPU takes the runs for its lowest energies; a call of high energies does not; both
    equal the oracle on a few directions. The setting can be taken back."""
    tr = I.weak_undulator(1000.0, 0.5e-10, 10e-6, 5, 4096)
    hw = I.omega_linear(128, 1.2 * I.undulator_first_harmonic_eV(1000.0, 0.5e-10, 10e-6))
    for k, some in ((1.0, True), (3e4, False)):
        grid = I.make_grid(hw * k, 32, 32, 2e-3)
        inp = rad.DeviceInputs(tr, grid)
        p, _ = plan_of(inp, rad.RAD_CLASSICAL, form)
        if form == rad.RAD_MIXED:
            assert p.set_phase_budget(1e9) == rad.RAD_OK
        got = cube_of(p, inp)
        assert (p.last_cut() > 0) == some, (k, p.last_cut())
        assert p.set_cut(0) == rad.RAD_OK and "cut=0" in p.describe().split()
        cube_of(p, inp)
        assert p.last_cut() == 0
        assert p.set_cut(-1) == rad.RAD_OK
        assert np.array_equal(cube_of(p, inp), got)
        if some:
            pick = np.arange(0, 1024, 97)
            sub = I.Grid(hw, grid.theta_x[pick].copy(), grid.theta_y[pick].copy(), grid.d_omega[pick].copy())
            ref = O.spectrum_cube(tr, sub, O.CLASSICAL)
            (assert_mixed_close if form == rad.RAD_MIXED else assert_fp64_close)(got[:, pick], ref)
        p.close()


def test_refused_settings():
    tr = bunch([300, 40])
    inp = rad.DeviceInputs(tr, directions(33, I.omega_log(200, 1e5, 4e8)))
    p, gran = plan_of(inp, rad.RAD_SPIN_HALF, rad.RAD_FP64)
    before = p.describe()
    with pytest.raises(rad.RadError):
        p.last_cut()  # nothing ran yet
    for bad in (-2, 1, gran - 1, inp.n_omega - 1, inp.n_omega + 1):
        assert p.set_cut(bad) == rad.RAD_EINVAL, bad
    assert p.describe() == before
    assert p.set_shape(1, 8, 64, 1) == rad.RAD_OK  # another shape is the direct kernel alone
    assert p.set_cut(inp.n_omega) == rad.RAD_EINVAL
    few = rad.DeviceInputs(tr, directions(15, I.omega_log(200, 1e5, 4e8)))
    q, _ = plan_of(few, rad.RAD_SPIN_HALF, rad.RAD_FP64)
    assert q.set_cut(few.n_omega) == rad.RAD_EINVAL


@pytest.mark.parametrize("mode", [rad.RAD_CLASSICAL, rad.RAD_SPIN_HALF])
@pytest.mark.parametrize("n_omega", [600, 640])
def test_double_float_energies_above_the_cut(mode, n_omega):
    """k_df starts at the cut and takes one or two energies per lane by how many 128s are left above it: every number of them
    from five down."""
    tr, grid = bunch([300, 41]), directions(17, I.omega_log(n_omega, 1e5, 5e8))
    ref = O.spectrum_cube(tr, grid, MODE_ORC[mode])
    inp = rad.DeviceInputs(tr, grid)
    p, _ = plan_of(inp, mode, rad.RAD_FP64_DF)
    for cut in range(0, n_omega, 128):
        assert p.set_cut(cut) == rad.RAD_OK
        assert_fp64_close(cube_of(p, inp), ref)
        assert p.last_cut() == cut
    p.close()
