"""The library's host side over a fake CUDA runtime (fake_cudart.c): entry
points run to their end without a GPU, their launches are recorded, and a
launch that a device would refuse fails."""
from __future__ import annotations

import ctypes
import os
import re
import subprocess

from paper_1804_02883_gb300 import binding
from paper_1804_02883_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
PTR = 1 << 40  # stands for device memory: aligned, never touched


class FakeRuntime:
    def __init__(self, out: str):
        B.build()
        objs = [os.path.join(B.OUT, s.replace(".cu", ".o")) for s in B.SOURCES]
        fake, so = os.path.join(out, "fake.o"), os.path.join(out, "libepd_lb_fake.so")
        inc = os.path.join(os.path.dirname(os.path.dirname(B.nvcc())), "include")
        subprocess.run(["gcc", "-O1", "-fPIC", "-w", f"-I{inc}", "-c", os.path.join(HERE, "fake_cudart.c"), "-o", fake], check=True)
        # (symbols bound inside the library: a CUDA runtime loaded beside it stays out of the way)
        subprocess.run([B.nvcc(), *B.ARCH, "-cudart", "none", "-shared", "-Xlinker", "-Bsymbolic", "-o", so, fake, *objs], check=True)
        self.L = L = ctypes.CDLL(so)
        L.fake_launch.restype = ctypes.c_char_p
        L.epd_lb_init.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p]
        L.epd_lb_destroy.argtypes = [ctypes.c_void_p]
        L.epd_prop_solve.argtypes = [ctypes.c_void_p] * 5 + [ctypes.c_size_t, ctypes.c_void_p]
        L.epd_sur_forward.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p, ctypes.c_double, ctypes.c_double] + \
            [ctypes.c_void_p] * 3 + [ctypes.c_size_t, ctypes.c_void_p]
        L.epd_sur_gradients.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p, ctypes.c_double, ctypes.c_double] + \
            [ctypes.c_void_p] * 5 + [ctypes.c_size_t, ctypes.c_void_p]
        L.epd_prop_solve3d.argtypes = [ctypes.c_void_p, ctypes.c_int32] + [ctypes.c_void_p] * 4 + [ctypes.c_size_t, ctypes.c_void_p]

    def init(self, runs):
        """(return code of epd_lb_init, its launches); the handle is released."""
        self.L.fake_reset()
        h = ctypes.c_void_p()
        rc = self.L.epd_lb_init(binding._params_array(runs), len(runs), None, 0, None, ctypes.byref(h))
        out = self.launches()
        if not rc:
            self.L.epd_lb_destroy(h)
        return rc, out

    def step_exact(self, runs, iterations):
        """(return code of one exact step of that many iterations, its launches)."""
        h = ctypes.c_void_p()
        rc = self.L.epd_lb_init(binding._params_array(runs), len(runs), None, 0, None, ctypes.byref(h))
        rc = rc or self.L.epd_lb_set_inversion(h, iterations, ctypes.c_double(0.0))
        self.L.fake_reset()
        rc = rc or self.L.epd_lb_step(h, ctypes.c_int64(1))
        out = self.launches()
        self.L.epd_lb_destroy(h)
        return rc, out

    def solve(self, run):
        self.L.fake_reset()
        n = ctypes.c_size_t()
        assert self.L.epd_prop_solve_workspace_bytes(ctypes.byref(run.c()), ctypes.byref(n)) == 0
        return self.L.epd_prop_solve(ctypes.byref(run.c()), PTR, PTR, PTR, PTR, n, None)

    def solve3d(self, run, nz):
        self.L.fake_reset()
        n = ctypes.c_size_t()
        assert self.L.epd_prop_solve3d_workspace_bytes(ctypes.byref(run.c()), nz, ctypes.byref(n)) == 0
        return self.L.epd_prop_solve3d(ctypes.byref(run.c()), nz, PTR, PTR, PTR, PTR, n, None)

    def sur_forward(self, run, batch):
        self.L.fake_reset()
        n = ctypes.c_size_t()
        assert self.L.epd_sur_workspace_bytes(run.ny, run.nx, batch, 0, ctypes.byref(n)) == 0
        return self.L.epd_sur_forward(ctypes.byref(run.c()), batch, PTR, 1.0, 1.0, PTR, PTR, PTR, n, None)

    def sur_gradients(self, run, batch):
        self.L.fake_reset()
        n = ctypes.c_size_t()
        assert self.L.epd_sur_workspace_bytes(run.ny, run.nx, batch, 1, ctypes.byref(n)) == 0
        return self.L.epd_sur_gradients(ctypes.byref(run.c()), batch, PTR, 1.0, 1.0, PTR, PTR, PTR, PTR, PTR, n, None)

    def launches(self):
        """(mangled kernel name, integral template arguments, grid, block, shared memory, cluster) of every launch."""
        out = []
        for i in range(self.L.fake_launches()):
            v = (ctypes.c_int * 6)()
            name = self.L.fake_launch(i, v).decode()
            args = tuple(int(a) for a in re.findall(r"L[ib](\d+)E", name))
            out.append((name, args, tuple(v[:3]), v[3], v[4], v[5]))
        return out
