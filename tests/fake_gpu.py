"""The library's host code linked against tests/fake_cudart.cpp: plans can be made, described and executed without a device.
Used through `plan`, in processes of their own (the fake's symbols are CUDA's)."""
import ctypes
import os
import subprocess
import sys

import paper_1910_10391_gb300.build as B

HERE = os.path.dirname(os.path.abspath(__file__))
PTR = ctypes.c_void_p(1 << 20)  # stands for device memory; the fake never follows it


def library(tmp):
    """Compile and link it into tmp (the library's own objects are compiled where they are missing or old)."""
    B.build()
    objs = []
    for s in B.SOURCES:
        obj, src = os.path.join(B.BUILD_DIR, s.replace(".cu", ".o")), os.path.join(B.CSRC, s)
        if not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(d) for d in B._deps()):
            obj = os.path.join(tmp, s.replace(".cu", ".o"))
            subprocess.check_call([B._nvcc()] + B.NVCC_FLAGS + ["-c", src, "-o", obj])
        objs.append(obj)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B._nvcc()))), "include")
    out = os.path.join(tmp, "librad_fake.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-I", inc, os.path.join(HERE, "fake_cudart.cpp")] +
                          objs + ["-o", out, "-Wl,-Bsymbolic", "-Wl,-z,lazy"])
    return out


class Fake:
    def __init__(self, path):
        self.lib = lib = ctypes.CDLL(path)
        i64, P = ctypes.c_int64, ctypes.c_void_p
        lib.rad_plan_create.argtypes = [i64] * 4 + [ctypes.c_int] * 3 + [ctypes.c_int32, ctypes.POINTER(P)]
        lib.rad_plan_execute.argtypes = [P] * 14 + [ctypes.c_int, P]
        lib.rad_plan_autotune.argtypes = [P] * 14 + [ctypes.c_int, P]
        lib.rad_plan_describe.argtypes = [P, ctypes.c_char_p, ctypes.c_int]
        lib.rad_plan_kernel_launches.argtypes = lib.rad_plan_destroy.argtypes = [P]
        lib.rad_plan_set_cut.argtypes = [P, i64]
        lib.rad_plan_set_shape.argtypes = [P] + [ctypes.c_int] * 4
        lib.fake_capacity.argtypes = [ctypes.c_size_t]
        lib.fake_used.restype = lib.fake_peak.restype = ctypes.c_size_t
        lib.fake_launches.argtypes = [ctypes.c_char_p, ctypes.c_int]

    def plan(self, samples, particles, omega, angles, mode, precision, want=1, n_bins=0):
        h = ctypes.c_void_p()
        rc = self.lib.rad_plan_create(samples, particles, omega, angles, mode, precision, want, n_bins, ctypes.byref(h))
        return rc, h

    def describe(self, h):
        buf = ctypes.create_string_buffer(512)
        self.lib.rad_plan_describe(h, buf, 512)
        return dict(kv.split("=") for kv in buf.value.decode().split())

    def args(self):
        return [PTR] * 9 + [PTR, None, None, None]

    def launches(self, h):
        """Kernels that one execute launches, by the count of the library and by the fake's."""
        self.lib.fake_launches(b"", 1)
        assert self.lib.rad_plan_execute(h, *self.args(), 0, None) == 0
        return self.lib.rad_plan_kernel_launches(h), self.lib.fake_launches(b"", 0)


def run(path, code):
    """Run code (with `f`, a Fake) in a process of its own."""
    src = f"import sys; sys.path[:0] = [{HERE!r}, {os.path.dirname(HERE)!r}]\nfrom fake_gpu import Fake\nf = Fake({path!r})\n" + code
    r = subprocess.run([sys.executable, "-c", src], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
