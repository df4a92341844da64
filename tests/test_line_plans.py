"""The radix plans of the in-place transforms (line_plan), called on the host:
every length has one of radices that the passes are built for, and the grids of
the GPU tests between them run every radix that any length takes."""
import ctypes

import pytest

import paper_1804_02883_gb300 as P
from test_gpu_line_plans import BOX, MORE
from test_gpu_lines import GRIDS

BOXES = [(2, 8, 8)]  # of test_gpu_solve3d.py

FIRST, INNER, LAST = {2, 4, 6, 8, 10, 12}, {3, 4, 5, 8, 9}, {1, 2, 3, 4, 5, 8, 9, 10, 15, 16}


class Plan(ctypes.Structure):
    _fields_ = [("w", ctypes.c_ulonglong), ("nf", ctypes.c_int)]


def plan(n, sites, fp64):
    f = P.lib()._ZN5epdlb9line_planEixb
    f.restype, f.argtypes = Plan, [ctypes.c_int, ctypes.c_longlong, ctypes.c_bool]
    p = f(n, sites, fp64)
    return [(p.w >> (8 * i)) & 255 for i in range(p.nf)]


def lengths():
    for n in range(2, 2049, 2):  # z axes start at 2, x and y at 8
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            yield n


def used(plans):
    return {"first": {p[0] for p in plans}, "inner": {r for p in plans for r in p[1:-1]}, "last": {p[-1] for p in plans}}


@pytest.mark.parametrize("fp64", [False, True])
def test_every_length_has_a_plan_that_a_test_runs(fp64):
    # the plan depends on the sites through three sizes of grid
    edges = [1 << 15, (1 << 20) - 1] if fp64 else [1 << 14]
    plans = []
    for n in lengths():
        for sites in [8 * n] + [s for e in edges for s in (e, e + 1) if s >= 8 * n]:
            p = plan(n, sites, fp64)
            prod = 1
            for r in p:
                prod *= r
            assert prod == n and 2 <= len(p) <= 4, (n, sites, p)
            assert p[0] in FIRST and p[-1] in LAST and set(p[1:-1]) <= INNER, (n, sites, p)
            plans.append(p)
    ran = [plan(n, ny * nx, fp64) for ny, nx in GRIDS + MORE for n in (ny, nx)]
    ran += [plan(n, ny * nx * nz, fp64) for nz, ny, nx in BOXES for n in (nz, ny, nx)]
    if fp64:
        ran += [plan(n, BOX[0] * BOX[1] * BOX[2], fp64) for n in BOX]
    want, got = used(plans), used(ran)
    for k in want:
        assert want[k] == got[k], k
