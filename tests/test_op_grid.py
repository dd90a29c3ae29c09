"""Block decomposition of the FP64 operator passes (csrc/op64.cu, op_shape), on the CPU: the tiles
and chunks cover the grid within the threads of a block, and a batch's work items, which name a
block by three 16-bit coordinates, hold it for cross sections of any size a context accepts."""
import ctypes
import re
import subprocess

import pytest

from paper_1302_3663_gb300 import bfibm

from test_cluster_layout import Geo


class OpShape(ctypes.Structure):
    _fields_ = [(f, ctypes.c_int) for f in "TX TY KC nx ny nc".split()]


class Dim3(ctypes.Structure):
    _fields_ = [(f, ctypes.c_uint) for f in "x y z".split()]


def function(name, restype, arg):
    bfibm.lib()
    out = subprocess.run(["nm", "-D", "--defined-only", bfibm.library_path()],
                         capture_output=True, text=True, check=True).stdout
    f = getattr(bfibm.lib(), re.search(r"\S*%s\S*" % name, out).group())
    f.restype, f.argtypes = restype, [ctypes.POINTER(arg)]
    return f


@pytest.mark.parametrize("n", [(2, 2, 2), (3, 5, 2), (17, 200, 40), (321, 18, 6), (128, 128, 256),
                               (160, 160, 320), (513, 33, 130), (4096, 4096, 4), (8192, 8192, 2),
                               (30000, 1200, 2), (2, 200000, 4), (20000, 2, 40), (600, 600, 1200)])
def test_items_hold_every_block(n):
    g = Geo(open=-1, h=1.0)
    for a in range(3):
        g.n[a], g.s[a] = n[a], n[a] + 1
    S = function("op_shape", OpShape, Geo)(ctypes.byref(g))
    d = function("op_grid3", Dim3, OpShape)(ctypes.byref(S))
    assert (S.TX + 2) * (S.TY + 2) <= 512
    assert S.nx * S.TX >= n[0] and S.ny * S.TY >= n[1] and S.nc * S.KC >= n[2]
    assert d.x * d.y * d.z == S.nx * S.ny * S.nc < 2 ** 31
    assert max(d.x, d.y, d.z) <= 65535
