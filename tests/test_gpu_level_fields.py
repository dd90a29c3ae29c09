"""The multigrid fields of every level after a solve, as the operator-level access shows them: the
cluster V-cycle (csrc/cluster.cu) leaves each level's iterate, right-hand side and residual in
global memory as a launch per phase does. (The coarsest pressure level's right-hand side may keep
the mean that its solve takes off.)"""
import numpy as np
import pytest

from paper_1302_3663_gb300 import bfibm

from helpers import cell_mask, face_mask
from test_gpu_cluster import FP64_TOL
from test_gpu_op64 import context

pytestmark = pytest.mark.gpu


def fields(n, per, tail, precision):
    c = context(n, per, 6, precision=precision)
    c.set_option(bfibm.OPT_TAIL, tail)
    c.solve_viscous(1)
    c.solve_pressure(1)
    get = c.get_field_f32 if precision else c.get_field
    out = []
    for l in range(1, c.levels):
        for d in range(c.dim):
            m = face_mask(c, d, l)
            for name in ("ut", "urhs") + (("ures",) if l < c.levels - 1 else ()):
                out.append(((l, name, d), get(name, d, l)[m]))
        m = cell_mask(c, l)
        for name in ("p", "prhs") + (("pres",) if l < c.levels - 1 else ()):
            a = get(name, 0, l)[m]
            if name == "prhs" and l == c.levels - 1:
                a = a - a.mean()
            out.append(((l, name, 0), a))
    c.close()
    return out


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,per", [((16, 16, 32), (0, 0, 1)), ((32, 48, 32), (1, 0, 1)),
                                   ((64, 32), (1, 0))])
def test_every_level_as_by_launches(n, per, precision):
    # one cycle: FP64 rounds otherwise in the launches (its residual's form), FP32 does not
    for (what, a), (_, b) in zip(fields(n, per, 1 << 20, precision), fields(n, per, 0, precision)):
        tol = 2.0 ** -22 if precision and what[1] == "prhs" else 0.0 if precision else FP64_TOL
        assert np.abs(a - b).max() <= tol * np.abs(b).max(), what
