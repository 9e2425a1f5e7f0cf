"""The calls that a user of this library has it do, as cases to be measured.

A case is a dict of plain values with a "kind":

  spectrum  photon spectra of an ensemble (rad_spectrum): cube, spectrum, radial bins
  labels    per-particle radial-bin spectra and their logarithms, the surrogate's training set
  planar    trajectories in the Doyle-Turner planar potential (rad_crystal_trajectories)
  axial     trajectories in the Doyle-Turner string potential (rad_axial_trajectories)
  train     training steps of the surrogate network, its weights and its predictions

`listed()` holds the workloads of this repository at their own sizes, or cut in particles, samples
or directions so that one pass stays below a second; `draw(rng)` gives others of the same ranges.
The mixed-precision form computes its sin/cos, its integrand and its sums in FP32 and leaves
results good to single precision in FP64 storage: a program that asks for that form keeps
them in single precision, and so does `run`.
"""
import math

import numpy as np
import torch

import paper_1910_10391_gb300 as rad
from paper_1910_10391_gb300 import inputs as I

HBARC, ALPHA, ME = 1.973269804e-7, 7.2973525693e-3, 0.51099895e6
R0, A0 = 2.8179403262e-15, 5.29177210903e-11
PRECISION = {"fp64": rad.RAD_FP64, "fp64_df": rad.RAD_FP64_DF, "mixed": rad.RAD_MIXED}
MODE = {"classical": rad.RAD_CLASSICAL, "spin0": rad.RAD_SPIN0, "spin_half": rad.RAD_SPIN_HALF}
# terms of the sum that a drawn case may have at most, by precision
MOST_TERMS = {"fp64": 4e9, "fp64_df": 3e10, "mixed": 6e11}
# terms up to which the plain 64-bit sum takes some seconds
EXACT_TERMS = 2.5e10


def listed():
    return [
        # one analytic trajectory on a small grid, the paper's precision: a first look at a spectrum
        dict(name="undulator_fp64", kind="spectrum", source="undulator", precision="fp64", mode="classical",
             particles=1, samples=4096, n_omega=128, n_side=16, out="cube"),
        # the same in the chosen form: the smallest call, latency and launches count
        dict(name="undulator_mixed", kind="spectrum", source="undulator", precision="mixed", mode="classical",
             particles=1, samples=4096, n_omega=128, n_side=16, out="cube"),
        # the paper's integral test: one long trajectory, many photon energies, odd sizes
        dict(name="strong_undulator_df", kind="spectrum", source="strong", precision="fp64_df", mode="classical",
             particles=1, samples=40961, n_omega=500, n_side=15, out="cube"),
        # an energy-losing beam cut into sections with their own energies, the paper's precision
        dict(name="sections_fp64", kind="spectrum", source="sections", precision="fp64", mode="spin_half",
             particles=8, samples=4000, n_omega=192, n_side=18, out="cube+spectrum"),
        # a slice of the positron ensemble at full accuracy
        dict(name="ensemble_df", kind="spectrum", source="ensemble", precision="fp64_df", mode="spin_half",
             particles=6, samples=12000, n_omega=384, n_side=24, out="cube+spectrum"),
        # one batch of the positron ensemble, the headline workload and the largest call
        dict(name="ensemble_mixed", kind="spectrum", source="ensemble", precision="mixed", mode="classical",
             particles=32, samples=20000, n_omega=512, n_side=64, out="cube"),
        # electrons of uneven lengths (2000 to 200000 samples): spectrum and radial bins only
        dict(name="batch_mixed", kind="spectrum", source="batch", precision="mixed", mode="spin_half",
             particles=64, samples=20000, n_omega=1024, n_side=24, out="spectrum+bins"),
        # training labels of the surrogate: one beam's per-particle spectra in radial bins
        dict(name="labels_mixed", kind="labels", particles=64, samples=8192, n_omega=256, n_side=32, gamma=12000.0),
        # entry conditions to records with every part of the physics, FP64
        dict(name="planar_fp64", kind="planar", precision="fp64", physics="all", charge=1, particles=1024,
             samples=2000),
        # a larger beam in the FP32 form with double-float state
        dict(name="planar_fp32", kind="planar", precision="fp32", physics="ms", charge=1, particles=2048,
             samples=2500),
        # axial channeling, strings of the <110> axis
        dict(name="axial_fp64", kind="axial", physics="ms", charge=1, particles=512, samples=1000),
        # training of the surrogate's network and a look at its predictions
        dict(name="surrogate_train", kind="train", batch=1024, n_in=62, width=256, depth=3, n_out=2048, steps=24),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spectrum"] * 6 + ["labels", "planar", "axial", "train"])
    if kind == "spectrum":
        p = rng.choice(["fp64", "fp64_df", "mixed", "mixed"])
        src = rng.choice(["undulator", "strong", "ensemble", "ensemble", "sections", "batch"])
        c = dict(kind=kind, source=src, precision=p, mode=rng.choice(["classical", "spin0", "spin_half"]),
                 particles=1 if src in ("undulator", "strong") else _log(rng, 2, 64),
                 samples=_log(rng, 1000, 40000) if src in ("undulator", "strong") else _log(rng, 1000, 20000),
                 n_omega=_log(rng, 24, 1024), n_side=_log(rng, 6, 64),
                 out=rng.choice(["cube", "cube+spectrum", "spectrum+bins"]))
        if src in ("undulator", "strong"):
            c["mode"] = "classical"
        while _terms(c) > MOST_TERMS[p]:
            k = rng.choice(["particles", "samples", "n_omega", "n_side"])
            c[k] = max(c[k] * 2 // 3, {"particles": 1, "samples": 1000, "n_omega": 24, "n_side": 6}[k])
        return c
    if kind == "labels":
        return dict(kind=kind, particles=_log(rng, 8, 96), samples=_log(rng, 1000, 8192), n_omega=_log(rng, 64, 256),
                    n_side=2 * rng.randint(6, 16), gamma=float(_log(rng, 2000, 40000)))
    if kind == "planar":
        return dict(kind=kind, precision=rng.choice(["fp64", "fp32"]), physics=rng.choice(["none", "ms", "all"]),
                    charge=rng.choice([1, -1]), particles=_log(rng, 30, 8192), samples=_log(rng, 100, 2000))
    if kind == "axial":
        return dict(kind=kind, physics=rng.choice(["none", "ms", "all"]), charge=rng.choice([1, -1]),
                    particles=_log(rng, 30, 2048), samples=_log(rng, 100, 1000))
    return dict(kind=kind, batch=_log(rng, 64, 1024), n_in=rng.choice([3, 20, 62]), width=32 * rng.randint(2, 8),
                depth=rng.randint(2, 4), n_out=2 * _log(rng, 32, 1024), steps=rng.randint(4, 24))


def _terms(c):
    """Terms of the sum over samples, photon energies and directions (mean lengths)."""
    return c["particles"] * (c["samples"] * (1.35 if c.get("source") == "batch" else 1.0)) * c["n_omega"] * c["n_side"] ** 2


# --------------------------------------------------------------------------- inputs
def _beam(case, seed):
    """Trajectories, grid and radial bins (host) of a spectrum case."""
    n, L, no, ns, src = case["particles"], case["samples"], case["n_omega"], case["n_side"], case["source"]
    rng = np.random.default_rng(seed)
    if src == "undulator":  # amplitude 0.3 to 0.6 A, 4 to 6 periods
        a, lam, g = rng.uniform(0.3, 0.6) * 1e-10, 10e-6, 1000.0
        tr = I.weak_undulator(g, a, lam, int(rng.integers(4, 7)), L)
        grid = I.make_grid(I.omega_linear(no, 1.2 * I.undulator_first_harmonic_eV(g, a, lam)), ns, ns, 2.0 / g)
    elif src == "strong":  # 2 GeV, 53 mm period, about 1 T, 0 to 500 eV within 5/gamma
        g = 2.0e9 / I.ME_EV
        tr = I.planar_undulator(g, I.undulator_K(rng.uniform(0.9, 1.1), 0.053), 0.053, 20, max(L // 20, 50))
        grid = I.make_grid(I.omega_linear(no, 500.0), ns, ns, 5.0 / g)
    elif src == "ensemble":
        tr, grid = I.channeling(n, 10e9, +1, L, 5e-9, seed), I._ensemble_grid(10e9, 20.0, no, ns)
    elif src == "sections":
        tr = I.channeling_sections(n, 10e9, +1, L, 5e-9, seed, 500).traj
        grid = I._ensemble_grid(10e9, 20.0, no, ns)
    else:  # lognormal lengths
        lens = I.lognormal_lengths(n, seed, median=L, lo=max(L // 10, 2), hi=10 * L)
        tr, grid = I.channeling(n, 20e9, -1, lens, 5e-9, seed), I._ensemble_grid(20e9, 20.0, no, ns)
    boa = I.radial_bins(grid.theta_x, grid.theta_y, 8, float(np.abs(grid.theta_x).max()) * 1.0001)
    return tr, grid, boa


def _label_beam(case, seed):
    """One beam of surrogate entries (scattering-free positrons of one Lorentz factor) on the
    theta_y > 0 half of the grid."""
    n, L, no, ns, g = case["particles"], case["samples"], case["n_omega"], case["n_side"], case["gamma"]
    rng = np.random.default_rng(seed)
    E = g * I.ME_EV
    thL = math.sqrt(2.0 * 20.0 / E)
    tmax = thL + 3.0 / g
    d = 2.0 * tmax / ns
    tx, ty = np.meshgrid(-tmax + (np.arange(ns) + 0.5) * d, (np.arange(ns // 2) + 0.5) * d, indexing="xy")
    tx, ty = np.ascontiguousarray(tx.ravel()), np.ascontiguousarray(ty.ravel())
    grid = I.Grid(I.omega_log(no, 1e-4 * E, 0.5 * E), tx, ty, np.full(tx.size, 2.0 * d * d))
    tr = I.channeling_given(rng.uniform(0, I.SI110_DP, n), rng.uniform(-1.5, 1.5, n) * thL, np.full(n, g), L,
                            100e-6 / 8191, ms=False)
    tr.weight = np.ones(n)
    return tr, grid, I.radial_bins(tx, ty, 8, tmax)


FLAGS = {"none": 0, "ms": rad.RAD_TRAJ_MS,
         "all": rad.RAD_TRAJ_MS | rad.RAD_TRAJ_MS_EL | rad.RAD_TRAJ_LL | rad.RAD_TRAJ_MS_LOSS}
FIELDS = ("t", "x", "y", "dz", "vx", "vy", "dvz", "ax", "ay", "az")


def _entries(case, seed):
    """Entry positions and angles of a trajectory case (host)."""
    n, rng = case["particles"], np.random.default_rng(seed)
    if case["kind"] == "planar":
        thL = math.sqrt(2.0 * 20.0 / 10e9)
        return rng.uniform(0, I.SI110_DP, n), None, rng.normal(0, 0.3 * thL, n), None
    psi = math.sqrt(2.0 * 35.0 / 10e9)
    a = 5.431e-10
    return rng.uniform(0, a, n), rng.uniform(0, a / math.sqrt(2.0), n), rng.normal(0, 0.3 * psi, n), rng.normal(0, 0.3 * psi, n)


def _train_data(case, seed):
    """Weights, minibatches, targets, masks and a held-out batch of a training case (GPU, FP32)."""
    B, k, W, D, O, S = (case[x] for x in ("batch", "n_in", "width", "depth", "n_out", "steps"))
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    new = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    x, xv = torch.tanh(new(S, B, k)), torch.tanh(new(B, k))
    t = torch.sin(x @ new(k, O) * (2.0 / math.sqrt(k)))
    mask = (torch.rand(S, B, O, generator=g, device="cuda") > 0.1).float()
    dims, parts = [k] + [W] * D + [O], []
    for a, b in zip(dims[:-1], dims[1:]):
        parts += [(torch.rand(b * a, generator=g, device="cuda") * 2 - 1) / math.sqrt(a), torch.zeros(b, device="cuda")]
    return torch.cat(parts), dims, x, t, mask, xv


# --------------------------------------------------------------------------- prepare and run
def _dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a)).to(dtype).to("cuda")


def prepare(case, seed):
    kind = case["kind"]
    f64 = dict(dtype=torch.float64, device="cuda")
    if kind == "spectrum":
        tr, grid, boa = _beam(case, seed)
        bins = "bins" in case["out"]
        inp = rad.DeviceInputs(tr, grid, bin_of_angle=boa if bins else None, n_bins=8 if bins else 0)
        return dict(kind=kind, inp=inp, mode=MODE[case["mode"]], precision=PRECISION[case["precision"]],
                    cube=torch.empty(inp.n_omega, inp.n_angles, **f64) if "cube" in case["out"] else None,
                    spectrum=torch.empty(inp.n_omega, **f64) if "spectrum" in case["out"] else None,
                    bins=torch.empty(inp.n_omega, 8, **f64) if bins else None)
    if kind == "labels":
        tr, grid, boa = _label_beam(case, seed)
        inp = rad.DeviceInputs(tr, grid, bin_of_angle=boa, n_bins=8)
        plan = rad.Plan(inp.n_samples, inp.n_particles, inp.n_omega, inp.n_angles, rad.RAD_SPIN_HALF, rad.RAD_MIXED,
                        rad.RAD_PER_PARTICLE | 4, 8)
        plan.set_phase_budget(65536.0)
        return dict(kind=kind, inp=inp, plan=plan, bins=torch.empty(inp.n_particles, inp.n_omega, 8, **f64),
                    labels=torch.empty(inp.n_particles, inp.n_omega, 8, dtype=torch.float32, device="cuda"))
    if kind in ("planar", "axial"):
        n, L = case["particles"], case["samples"]
        flags = FLAGS[case["physics"]] | (rad.RAD_TRAJ_FP32 if case.get("precision") == "fp32" else 0)
        ch = rad.RadChannel(0.0, I.SI110_DP, I.EPS_S_EV, I.SI_X0, I.RHO_THERMAL, I.ME_EV, case["charge"], flags)
        fit = (I.SYNTH_DT_AX, I.SYNTH_DT_BX, I.SYNTH_DT_CX, I.SI_I_EV)
        if kind == "planar":
            pot = rad.RadPlanarPotential.make(I.SYNTH_DT_A, I.SYNTH_DT_B, I.SI_N, *fit, n_neighbours=3)
        else:
            pot = rad.RadAxialPotential.make(I.SYNTH_DT_A, I.SYNTH_DT_B,
                                             rad.crystal_string_lattice(rad.RAD_DIAMOND, 5.431e-10, 110), *fit, n_cells=2)
        return dict(kind=kind, ch=ch, pot=pot, seed=int(seed) % (1 << 31),
                    off=torch.arange(n + 1, dtype=torch.int64, device="cuda") * L, energy=torch.full((n,), 10e9, **f64),
                    entry=[None if v is None else _dev(v) for v in _entries(case, seed)], out=torch.empty(n * L, 10, **f64))
    w, dims, x, t, mask, xv = _train_data(case, seed)
    net = rad.MLP(case["n_in"], case["width"], case["depth"], case["n_out"], max_batch=case["batch"], seed=1)
    net.set_params(w.cpu().numpy())
    return dict(kind=kind, net=net, x=x, t=t, mask=mask, xv=xv, y=torch.empty(case["batch"], case["n_out"], device="cuda"),
                loss=torch.zeros(case["steps"], device="cuda"))


def _ok(rc, where):
    if rc:
        raise rad.RadError(rc, where)


def run(state):
    s = state
    if s["kind"] == "spectrum":
        i, bins = s["inp"], s["bins"] is not None
        _ok(rad.rad_spectrum(*i.args(), s["mode"], s["precision"], s["cube"], s["spectrum"], i.boa if bins else None,
                             i.n_bins if bins else 0, s["bins"]), "rad_spectrum")
        out = {k: s[k] for k in ("cube", "spectrum", "bins") if s[k] is not None}
        return {k: v.float() for k, v in out.items()} if s["precision"] == rad.RAD_MIXED else out
    if s["kind"] == "labels":
        _ok(s["plan"].execute(*s["inp"].args(), None, None, s["inp"].boa, s["bins"]), "rad_plan_execute")
        rad._binding.rad_log_targets(s["bins"], 1e-30, s["labels"])
        return s["labels"]
    if s["kind"] == "planar":
        x0, _, th, _ = s["entry"]
        _ok(rad.rad_crystal_trajectories(s["ch"], s["pot"], s["off"], s["energy"], x0, th, s["out"], 5e-9, s["seed"]),
            "rad_crystal_trajectories")
        return dict(zip(FIELDS, s["out"].unbind(1)))
    if s["kind"] == "axial":
        x0, y0, th, thy = s["entry"]
        _ok(rad.rad_axial_trajectories(s["ch"], s["pot"], s["off"], s["energy"], x0, th, s["out"], 5e-9, s["seed"],
                                       y0=y0, thy0=thy), "rad_axial_trajectories")
        return dict(zip(FIELDS, s["out"].unbind(1)))
    net = s["net"]
    for k in range(s["x"].shape[0]):
        net.train_step(s["x"][k], s["t"][k], 1e-3, 1e-5, s["loss"][k:k + 1], s["mask"][k])
    net.forward(s["xv"], s["y"])
    return {"weights": net.get(0), "loss": s["loss"], "predictions": s["y"]}


def work(case):
    """Bytes: each input read once, each output written once. Operations: those of the sum as
    written (one phase product and two or three complex multiply-adds a term), of one force sum
    per stage, of the network's matrix products."""
    if case["kind"] in ("spectrum", "labels"):
        if case["kind"] == "labels":
            n_ang, mode = case["n_side"] ** 2 // 2, "spin_half"
            samples, out = case["particles"] * case["samples"], case["particles"] * case["n_omega"] * 8 * 12
        else:
            n_ang, mode = case["n_side"] ** 2, case["mode"]
            samples = int(_terms(case) / (case["n_omega"] * n_ang))
            out = 8 * case["n_omega"] * (n_ang if "cube" in case["out"] else 9)
        return {"bytes": samples * 80 + out, "flops": samples * case["n_omega"] * n_ang * (13 if mode == "spin_half" else 9)}
    n = case["particles"] * case["samples"] if case["kind"] != "train" else 0
    if case["kind"] == "planar":
        return {"bytes": n * 80, "flops": n * 4 * 24 * 20}
    if case["kind"] == "axial":
        return {"bytes": n * 80, "flops": n * 4 * 4 * 4 * 10 * 20}
    B, W, D, O, S = (case[x] for x in ("batch", "width", "depth", "n_out", "steps"))
    mac = B * (W * case["n_in"] + (D - 1) * W * W + W * O)
    par = W * case["n_in"] + (D - 1) * W * W + W * O
    return {"bytes": S * (28 * par + B * (4 * case["n_in"] + 8 * O)), "flops": 2 * mac * (3 * S + 1)}


# --------------------------------------------------------------------------- 64-bit results
def exact(case, seed):
    if case["kind"] == "spectrum":
        if _terms(case) > EXACT_TERMS:
            return None
        tr, grid, boa = _beam(case, seed)
        cube = sum(_cubes(tr, grid, case["mode"]))
        out = {}
        if "cube" in case["out"]:
            out["cube"] = cube
        if "spectrum" in case["out"]:
            out["spectrum"] = cube @ _dev(grid.d_omega)
        if "bins" in case["out"]:
            out["bins"] = _bins(cube, grid, boa)
        return out
    if case["kind"] == "labels":
        n_terms = case["particles"] * case["samples"] * case["n_omega"] * case["n_side"] ** 2 // 2
        if n_terms > EXACT_TERMS:
            return None
        tr, grid, boa = _label_beam(case, seed)
        return torch.stack([torch.log10(_bins(c, grid, boa).clamp(min=1e-30)) for c in _cubes(tr, grid, "spin_half")])
    if case["kind"] in ("planar", "axial"):
        if case["particles"] * case["samples"] > 6e6 and case["kind"] == "planar":
            return None
        return dict(zip(FIELDS, _trajectories(case, seed)))
    return _trained(case, seed)


def _bins(cube, grid, boa):
    boa, dom = torch.as_tensor(boa).to("cuda"), _dev(grid.d_omega)
    return torch.stack([cube @ (dom * (boa == b)) for b in range(8)], 1)


def _cubes(tr, grid, mode):
    """The weighted cube of each particle: the sum of Sec. II in the expanded form, in FP64."""
    hw, tx, ty = _dev(grid.hbar_omega_eV), _dev(grid.theta_x), _dev(grid.theta_y)
    for p in range(tr.n_particles):
        S = _dev(tr.samples[tr.offsets[p]:tr.offsets[p + 1]])
        t, x, y, dz, vx, vy, dvz, ax, ay, az = S.unbind(1)
        g, E, L = float(tr.gamma[p]), float(tr.energy_eV[p]), S.shape[0]
        w = torch.cat([t[1:2] - t[:1], t[2:] - t[:-2], t[-1:] - t[-2:-1]]) * 0.5
        u = hw / E
        ws = (hw / HBARC) / (1.0 - u) if mode != "classical" else hw / HBARC
        cube = torch.empty(hw.numel(), tx.numel(), dtype=torch.float64, device="cuda")
        nd = max(1, min(tx.numel(), int(4e7 // (hw.numel() * L))))
        kc = max(1, int(4e7 // (hw.numel() * nd)))
        for j in range(0, tx.numel(), nd):
            nx, ny = tx[j:j + nd, None], ty[j:j + nd, None]
            c = 1.0 / (2.0 * g * g) + (nx * nx + ny * ny) * 0.5
            A = ((c * t - dz) - nx * x) - ny * y
            D = c - dvz - nx * vx - ny * vy
            m = az + nx * ax + ny * ay
            gw = w / (D * D)
            a, b = nx - vx, ny - vy
            fx, fy = (a * m - ax * D) * gw, (b * m - ay * D) * gw
            f = torch.stack([fx, fy, -(nx * fx + ny * fy), m * gw], 2)  # transversality gives f_z
            amp = 0
            for k in range(0, L, kc):
                ph = ws[None, :, None] * A[:, None, k:k + kc]
                amp = amp + torch.complex(torch.cos(ph) @ f[:, k:k + kc], torch.sin(ph) @ f[:, k:k + kc])
            q = amp.real ** 2 + amp.imag ** 2
            I2 = q[..., :3].sum(-1)
            if mode == "spin0":
                I2 = (1.0 - u) * I2
            elif mode == "spin_half":
                I2 = 0.5 * (1.0 + (1.0 - u) ** 2) * I2 + u ** 2 / (2.0 * g * g) * q[..., 3]
            cube[:, j:j + nd] = I2.T
        yield cube * (float(tr.weight[p]) * ALPHA / (4.0 * math.pi ** 2))


def _normals(seed, ids, step):
    """Philox4x32-10 words of (id, step, 1, id high) under the key `seed`, two 53-bit uniforms, Box-Muller."""
    M = np.uint64(0xFFFFFFFF)
    c = [ids & M, np.full_like(ids, step), np.full_like(ids, 1), ids >> np.uint64(32)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & M, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & M]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    uni = lambda a, b: (((a >> np.uint64(5)) << np.uint64(26) | (b >> np.uint64(6))).astype(np.float64) + 0.5) * 2.0 ** -53  # noqa: E731
    u1, u2 = uni(c[0], c[1]), uni(c[2], c[3])
    r = np.sqrt(-2.0 * np.log(u1))
    return r * np.cos(2 * np.pi * u2), r * np.sin(2 * np.pi * u2)


def _trajectories(case, seed):
    """RK4 records of Sec. III in numpy, all particles at once: the ten fields, particle after particle."""
    n, L, q, dt, mass, rho = case["particles"], case["samples"], case["charge"], 5e-9, ME, I.RHO_THERMAL
    flags = FLAGS[case["physics"]]
    ms, el = flags & rad.RAD_TRAJ_MS, flags & rad.RAD_TRAJ_MS_EL
    ll, lossy = flags & rad.RAD_TRAJ_LL, flags & rad.RAD_TRAJ_MS_LOSS
    a, ax_ = np.array(I.SYNTH_DT_A), np.array(I.SYNTH_DT_AX)
    C = np.array(I.SYNTH_DT_B) / (4 * np.pi ** 2) + rho ** 2
    CX = np.array(I.SYNTH_DT_BX) / (4 * np.pi ** 2) + rho ** 2
    e2 = ALPHA * HBARC
    if case["kind"] == "planar":
        dp = I.SI110_DP
        kf = 2.0 * q * 2.0 * math.sqrt(math.pi) * e2 * A0 * I.SI_N * dp * a / C ** 1.5
        j = np.arange(-2, 4)

        def planes(x):
            return (x - np.floor(x / dp) * dp)[:, None] - j * dp

        def force(x, y):
            r = planes(x)[:, :, None]
            return (kf * r * np.exp(-r * r / C)).sum((1, 2)), 0.0

        def densities(x, y):
            r = planes(x)
            nuc = dp / (math.sqrt(math.pi) * rho) * np.exp(-r[:, 2:4] ** 2 / rho ** 2).sum(1)
            r = r[:, :, None]
            return nuc, (I.SI_N * dp / math.sqrt(math.pi) * ax_ / np.sqrt(CX) * np.exp(-r * r / CX)).sum((1, 2)) + I.SYNTH_DT_CX * I.SI_N * nuc
    else:
        lat = rad.crystal_string_lattice(rad.RAD_DIAMOND, 5.431e-10, 110)  # the geometry is an input here
        nb, Lx, Ly, d = lat.n_strings, lat.cell_x, lat.cell_y, lat.d
        sx, sy = np.array(lat.sx[:nb]), np.array(lat.sy[:nb])
        N = nb / (d * Lx * Ly)
        kf = q * (2.0 * e2 * A0 / d) * (a / C) * (2.0 / C)
        im = np.arange(-2, 3)

        def offsets(x, y):
            ux = (x - np.floor(x / Lx) * Lx)[:, None, None] - sx[:, None] - im * Lx
            uy = (y - np.floor(y / Ly) * Ly)[:, None, None] - sy[:, None] - im * Ly
            return ux[..., None], uy[..., None]

        def force(x, y):
            ux, uy = offsets(x, y)
            gx, gy = np.exp(-ux * ux / C), np.exp(-uy * uy / C)
            return (kf * (ux * gx).sum(2) * gy.sum(2)).sum((1, 2)), (kf * gx.sum(2) * (uy * gy).sum(2)).sum((1, 2))

        def densities(x, y):
            ux, uy = offsets(x, y)
            gauss = lambda k: np.exp(-ux * ux / k).sum(2) * np.exp(-uy * uy / k).sum(2)  # noqa: E731
            nuc = gauss(rho ** 2).sum((1, 2)) / (math.pi * rho ** 2 * N * d)
            return nuc, (ax_ / CX * gauss(CX)).sum((1, 2)) / (math.pi * d) + I.SYNTH_DT_CX * N * nuc

    llk = -(2.0 / 3.0) * e2 / mass ** 2
    x0, y0, tx, ty = _entries(case, seed)
    zero = np.zeros(n)
    s = [x0.copy(), zero if y0 is None else y0, tx, zero if ty is None else ty, zero, np.full(n, 10e9)]
    g0 = s[5] / mass
    beta0, q0 = 1.0 - 1.0 / (2.0 * g0 * g0), 1.0 / (4.0 * g0 ** 4)

    def deriv(s):
        g, vp2 = s[5] / mass, s[2] ** 2 + s[3] ** 2
        vz = np.sqrt(1.0 - 1.0 / (g * g) - vp2)
        dvz = ((g - g0) * (g + g0) / ((g * g) * (g0 * g0)) - vp2 - q0) / (vz + beta0)
        fx, fy = force(s[0], s[1])
        return [s[2], s[3], fx / s[5], fy / s[5] + zero, dvz, llk * g * g * (fx * fx + fy * fy) if ll else zero], vz

    key, ids = int(seed) % (1 << 31), np.arange(n, dtype=np.uint64)
    rec = np.empty((L, 10, n))
    kx = ky = zero
    for k in range(L):
        k1, vz = deriv(s)
        ax, ay, g = k1[2] + kx, k1[3] + ky, s[5] / mass
        az = (k1[5] / mass / g ** 3 - (s[2] * ax + s[3] * ay)) / vz
        rec[k] = [np.full(n, k * dt), s[0], s[1], s[4], s[2], s[3], k1[4], ax, ay, az]
        k2, _ = deriv([u + 0.5 * dt * v for u, v in zip(s, k1)])
        k3, _ = deriv([u + 0.5 * dt * v for u, v in zip(s, k2)])
        k4, _ = deriv([u + dt * v for u, v in zip(s, k3)])
        s = [u + dt / 6.0 * (p + 2 * r + 2 * v + w) for u, p, r, v, w in zip(s, k1, k2, k3, k4)]
        kx = ky = zero
        if ms:
            E, (nuc, nel) = s[5], densities(s[0], s[1])
            var = 0.5 * I.EPS_S_EV ** 2 * (dt / I.SI_X0) / (E * E) * nuc
            if el:
                g = E / mass
                b2 = 1.0 - 1.0 / (g * g)
                br = np.maximum(np.log(2.0 * ME / I.SI_I_EV * g * g * b2) - b2, 0.0)
                var = var + 0.5 * dt * math.pi * R0 ** 2 * nel * br / (g * g * b2 * b2)
            z0, z1 = _normals(key, ids, k)
            dx, dy = np.sqrt(var) * z0, np.sqrt(var) * z1
            kx, ky = dx / dt, dy / dt
            s[2], s[3] = s[2] + dx, s[3] + dy
            if lossy:
                s[5] = E - mass * ALPHA / (2 * np.pi) * (E / mass) ** 3 * (dx * dx + dy * dy)
    return [torch.from_numpy(np.ascontiguousarray(rec[:, f].T).ravel()) for f in range(10)]


def _trained(case, seed):
    """The same training in FP64: GELU (erf) network, masked mean-squared error, AdamW."""
    w, dims, x, t, mask, xv = _train_data(case, seed)
    w, x, t, mask, xv = (v.double() for v in (w, x, t, mask, xv))
    m, v, losses = torch.zeros_like(w), torch.zeros_like(w), []

    def net(w, h):
        at = 0
        for l, (a, b) in enumerate(zip(dims[:-1], dims[1:])):
            h = h @ w[at:at + a * b].view(b, a).T + w[at + a * b:at + a * b + b]
            at += a * b + b
            h = torch.nn.functional.gelu(h) if l < len(dims) - 2 else h
        return h

    for k in range(x.shape[0]):
        w.requires_grad_(True)
        loss = (mask[k] * (net(w, x[k]) - t[k]) ** 2).mean()
        (g,) = torch.autograd.grad(loss, w)
        with torch.no_grad():
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            w = w.detach() - 1e-3 * ((m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8) + 1e-5 * w.detach())
        losses.append(loss.detach())
    with torch.no_grad():
        return {"weights": w, "loss": torch.stack(losses), "predictions": net(w, xv)}
