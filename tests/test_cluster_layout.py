"""The shared-memory layout of the cluster V-cycle (csrc/cluster.cu, cl_bytes),
on the CPU: every array that the kernel indexes lies inside the bytes that the
launch asks for, no two overlap, and a right-hand side that the kernel rewrites
has a place there. Levels that barely fit are what goes wrong: the layout then
leaves the right-hand sides of its first level in global memory."""
import ctypes
import re
import subprocess

import pytest

from paper_1302_3663_gb300 import bfibm

SMEM = 227 * 1024   # of a thread block, at most
KMAX = 8            # levels
I3 = ctypes.c_int * 3


class Geo(ctypes.Structure):
    _fields_ = [("n", I3), ("s", I3), ("per", I3), ("st", ctypes.c_longlong * 3),
                ("h", ctypes.c_double), ("open", ctypes.c_int)]


class ClLv(ctypes.Structure):
    _fields_ = ([(f, ctypes.c_int) for f in "n0 R nS s0 sR RS CP PS nh".split()] +
                [(f, ctypes.c_uint) for f in "mnh mR ms0 msR".split()] +
                [(f, ctypes.c_int) for f in "C pc na last k0 npl lo hi nlo per0 perR perS "
                 "st1 st2 fs".split()] +
                [("u", I3), ("f", I3), ("g", I3), ("c", ctypes.c_int), ("e", I3),
                 ("gl", I3)])


def cl_bytes():
    bfibm.lib()
    out = subprocess.run(["nm", "-D", "--defined-only", bfibm.library_path()],
                         capture_output=True, text=True, check=True).stdout
    f = getattr(bfibm.lib(), re.search(r"\S*cl_bytes\S*", out).group())
    f.restype = ctypes.c_size_t
    f.argtypes = [ctypes.c_int, ctypes.c_bool, ctypes.c_bool, ctypes.POINTER(Geo)] + \
        [ctypes.c_int] * 4 + [ctypes.POINTER(ClLv)]
    return f


def levels(n, per):
    """The grids of the multigrid hierarchy, halved as bfibm_create does."""
    n, out = list(n), []
    while True:
        D = len(n)
        g = Geo(open=-1, h=1.0)
        for a in range(3):
            g.n[a] = n[a] if a < D else 1
            g.per[a] = per[a] if a < D else 1
            g.s[a] = g.n[a] + (0 if g.per[a] else 1)
        g.st[0], g.st[1] = 1, (g.s[0] + 7) // 8 * 8
        g.st[2] = g.st[1] * g.s[1]
        out.append(g)
        if len(out) == 6 or any(v % 2 for v in n) or min(n) < 4 or \
                any(p and v // 2 % 2 for v, p in zip(n, per)):
            return out
        n = [v // 2 for v in n]


GRIDS = [((100, 50, 100), (0, 0, 1)), ((90, 90, 64), (0, 0, 1)), ((66, 66, 132), (0, 0, 1)),
         ((604, 800), (1, 0)), ((64, 64, 64), (0, 0, 1)), ((144, 144, 288), (0, 0, 1)),
         ((101, 75, 130), (0, 0, 1)), ((30, 22, 26), (1, 0, 0)), ((50, 46, 50), (0, 0, 0)),
         ((22, 16), (1, 0)), ((6, 6, 6), (0, 0, 1)), ((256, 128), (1, 0)), ((301, 199), (0, 0)),
         ((40, 24, 44), (1, 1, 1)), ((1022, 34), (1, 0))]


@pytest.mark.parametrize("n,per", GRIDS)
def test_every_array_lies_inside_the_allocation(n, per):
    f, g = cl_bytes(), levels(n, per)
    L, D = len(g), len(n)
    arr = (Geo * KMAX)(*g)
    for fp64 in (False, True):
        for V in (False, True):
            for start in range(L):
                for C in (1, 2, 4, 8, 16):
                    lv = (ClLv * KMAX)()
                    b = f(D, fp64, V, arr, L, start, C, 0, lv)
                    assert b <= SMEM
                    if b:
                        check(lv, D, fp64, V, L, start, b)


def check(lv, D, fp64, V, L, start, total):
    spans = []
    for l in range(start, L):
        v, el = lv[l], 8 if fp64 or l == L - 1 else 4

        def add(off, first, planes):
            spans.append((el * (off + first * v.PS), el * (off + (first + planes) * v.PS)))
        for d in range(D if V else 1):
            add(v.u[d], 0, v.pc + 2)
        if V:
            add(v.c, 0, v.pc + 1)
            for q in range(3 if D == 3 else 1):
                add(v.e[q], 1, v.pc + (1 if D == 2 or q >= 1 else 0))
        else:
            for a in range(D):
                add(v.e[a], 1, v.pc + (1 if a == D - 1 else 0))
        if v.fs:
            for d in range(D if V else 1):
                add(v.f[d], 1, v.pc)
                if V or el == 8:
                    add(v.g[d], 1, v.pc)
                if el == 8:
                    add(v.gl[d], 1, v.pc)
        else:
            assert l == start and set(v.f) | set(v.g) | set(v.gl) == {-1}
        # the kernel writes these right-hand sides: the restricted one below the first level,
        # the converted one of a mixed cycle, the pressure's without its mean
        if l > start or (l == L - 1 and (not V or not fp64)):
            assert v.fs
    assert all(0 <= lo < hi <= total for lo, hi in spans)
    spans.sort()
    assert all(a[1] <= b[0] for a, b in zip(spans, spans[1:]))
