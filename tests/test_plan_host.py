"""Host side of plans without a device (fake_cudart.cpp): what they allocate, what they fall back to when memory is short."""
import pytest

import fake_gpu


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fake_gpu.library(str(tmp_path_factory.mktemp("fake")))


# samples, particles, energies, directions, model, precision (0 FP64, 2 double-float)
SHAPES = [(40961, 1, 512, 225, 0, 0), (40961, 1, 512, 225, 0, 2), (32000, 64, 192, 324, 2, 0), (72000, 6, 384, 576, 2, 2)]


@pytest.mark.parametrize("shape", SHAPES)
def test_short_memory_falls_back_to_the_direct_kernel(fake, shape):
    """The moment kernel's scratch or its finer split do not fit: the plan is the direct kernel's, with its split and nothing
    held for the moment kernel, wherever that plan fits."""
    out = fake_gpu.run(fake, f"""
shape = {shape}
def sizes(cut):
    rc, h = f.plan(*shape)
    assert rc == 0
    assert f.lib.rad_plan_set_cut(h, cut) == 0
    d = f.describe(h)
    f.launches(h)  # the library's own tables are there from now on
    f.lib.rad_plan_destroy(h)
    return d
route, direct = sizes(shape[2]), sizes(0)
assert route["cut"] != "0" and direct["cut"] == "0"
# what a plan of the direct kernel alone needs, from the least capacity that admits one
lo, hi = 0, 1 << 36
while hi - lo > 1:
    mid = (lo + hi) // 2
    f.lib.fake_capacity(mid)
    rc, h = f.plan(*shape)
    f.lib.rad_plan_destroy(h) if rc == 0 else None
    lo, hi = (lo, mid) if rc == 0 else (mid, hi)
least = hi
ncomp = 8 if shape[4] == 2 else 6
parts = int(direct["chunks"]) * shape[2] * shape[3] * (ncomp if direct["amp"] == "1" else 1) * 8
need = f.lib.fake_used() + parts + shape[2] * shape[3] * 8 + 4096
assert least <= need, (least, need)
seen = set()
for k in range(64):  # capacities up to beyond the moment kernel's needs
    f.lib.fake_capacity(least + k * (1 << 24))
    rc, h = f.plan(*shape)
    assert rc == 0
    d = f.describe(h)
    assert f.lib.fake_used() <= least + k * (1 << 24)
    if d["cut"] == "0":
        assert {{q: d[q] for q in ("chunks", "amp", "nq", "R")}} == {{q: direct[q] for q in ("chunks", "amp", "nq", "R")}}, (k, d, direct)
        assert f.lib.fake_used() <= need
    seen.add(d["cut"])
    n, m = f.launches(h)
    assert n == m, (n, m)
    f.lib.rad_plan_destroy(h)
    assert f.lib.fake_used() <= 1 << 20
print(sorted(seen), least, need)
""")
    print(out)


# samples, particles, energies, directions, model, precision: few work items, so that the moment or node kernel would leave
# most of the SMs idle, or too few energies for its fixed cost
SMALL = [(1478, 7, 80, 16, 2, 0), (1478, 7, 80, 33, 2, 2), (340, 2, 512, 16, 0, 0), (340, 2, 513, 16, 0, 2), (1031, 1, 130, 40, 2, 2),
         (1468, 4, 129, 25, 0, 1), (2999, 1, 160, 16, 2, 1), (512, 1, 96, 16, 0, 1), (4000, 2, 24, 16, 0, 0)]
LARGE = [(4096, 1, 128, 256, 0, 0), (4096, 1, 128, 256, 0, 1), (40961, 1, 500, 225, 0, 2), (32000, 64, 192, 324, 2, 0),
         (72000, 6, 384, 576, 2, 2), (640000, 32, 512, 4096, 0, 1), (524288, 64, 256, 512, 2, 1), (19200, 64, 512, 1024, 2, 1)]


def test_calls_that_cannot_gain_are_the_direct_kernels(fake):
    """Where the costs exclude the route whatever the trajectories, a plan has the direct kernel's split, memory and number
    of launches; the calls of the library's workloads keep the route."""
    fake_gpu.run(fake, f"""
for shape in {SMALL}:
    found = []
    for cut in (-1, 0):
        rc, h = f.plan(*shape)
        assert rc == 0
        assert f.lib.rad_plan_set_cut(h, cut) == 0
        d, n = f.describe(h), f.launches(h)
        assert n[0] == n[1]
        used = f.lib.fake_used()
        f.lib.rad_plan_destroy(h)
        found.append((d, n, used - f.lib.fake_used()))
    assert found[0] == found[1], (shape, found)
    assert found[0][0]["cut"] == "0"
for shape in {LARGE}:
    rc, h = f.plan(*shape)
    assert f.describe(h)["cut"] == "auto", shape
    n = f.launches(h)
    assert n[0] == n[1]
    f.lib.rad_plan_destroy(h)
""")


def test_double_float_energies_per_lane(fake):
    """Two energies per lane unless that leaves half of a block idle or the GPU unfilled: calls that stay with the direct
    kernel lose nothing to the moment kernel's granularity of 128."""
    fake_gpu.run(fake, """
for n, R in ((1, 1), (64, 1), (128, 1), (129, 2), (256, 2), (257, 1), (300, 1), (384, 1), (385, 2), (512, 2), (1024, 2), (1536, 2),
             (1537, 2), (1280 + 128, 1), (1664, 2)):
    for angles, samples, want in ((64, 4000, R), (4, 4000, R if n <= 256 else 1), (40, 400, R if n <= 256 else 1)):
        rc, h = f.plan(samples, 2, n, angles, 0, 2)
        assert rc == 0
        assert f.lib.rad_plan_set_cut(h, 0) == 0
        assert f.describe(h)["R"] == str(want), (n, angles, samples, f.describe(h))
        assert f.launches(h)[0] == f.launches(h)[1] == 3
        f.lib.rad_plan_destroy(h)
""")


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_autotune_times_the_current_choice_first(fake, precision):
    """A budget that ends with the first candidate keeps the plan as it is."""
    fake_gpu.run(fake, f"""
rc, h = f.plan(640000, 32, 512, 4096, 0, {precision})
assert rc == 0
before = f.describe(h)
assert before["cut"] == "auto"
assert f.lib.rad_plan_autotune(h, *f.args(), 0, None) == 0
assert f.describe(h) == before, (before, f.describe(h))
""")


def test_training_graphs_have_their_own_arguments(fake):
    """Steps of two batch sizes may be in flight on two streams: the graph of one must not find the other's pointers."""
    fake_gpu.run(fake, """
import ctypes
P, i64, c, fl = ctypes.c_void_p, ctypes.c_int64, ctypes.c_int, ctypes.c_float
f.lib.rad_mlp_create.argtypes = [c, c, c, c, i64, ctypes.c_uint64, ctypes.POINTER(P)]
f.lib.rad_mlp_train_step.argtypes = [P, P, P, P, i64, fl, fl, P, P]
f.lib.fake_set_args.restype = P
h, x = P(), P(1 << 20)
assert f.lib.rad_mlp_create(3, 66, 2, 34, 600, 1, ctypes.byref(h)) == 0
where = {}
for batch in [600] * 3 + [33] * 3 + [600, 33, 1, 1, 1, 2, 2, 2, 5, 5, 5, 600, 600, 600]:
    f.lib.fake_launches(b"", 1)
    assert f.lib.rad_mlp_train_step(h, x, x, None, batch, 1e-3, 0.0, None, None) == 0
    if f.lib.fake_launches(b"k_set_args", 0):
        where.setdefault(batch, set()).add(f.lib.fake_set_args())
assert set(where) == {600, 33, 1, 2, 5}, where
seen = [a for s in where.values() for a in s]
assert len(seen) == len(set(seen)) == 6, where  # 600 was replaced and built again, with arguments of its own
""")
