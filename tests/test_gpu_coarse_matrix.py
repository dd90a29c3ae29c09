"""The coarsest solve as a matrix (csrc/cluster.cu, k_coarse_matrix) against its sweeps on
coarsest levels that take the matrix: up to its row limits (384 with a fixed count of V-cycles,
800 to a tolerance) and just past them, walled and periodic axes in every place. A context made
for one V-cycle per solve keeps the sweeps; the device memory a context asks for tells which."""
import numpy as np
import pytest

from paper_1302_3663_gb300 import bfibm

from test_gpu_cluster import FP64_TOL
from test_gpu_op64 import context

pytestmark = pytest.mark.gpu

# grid, periodic axes, level limit, rows of the coarsest level (pressure, viscous)
CASES = [((8, 8, 16), (0, 0, 1), 2, 128, 384), ((10, 10, 12), (0, 0, 1), 6, 150, 450),
         ((14, 38, 4), (0, 0, 1), 6, 266, 798), ((4, 134, 4), (0, 0, 1), 6, 268, 804),
         ((20, 20, 16), (0, 0, 1), 2, 800, 2400), ((18, 10, 36), (0, 0, 1), 6, 810, 2430),
         ((12, 10, 8), (1, 0, 1), 2, 120, 360), ((8, 12, 10), (1, 1, 0), 2, 120, 360),
         ((8, 4, 20), (0, 1, 0), 6, 80, 240), ((4, 8, 12), (1, 1, 1), 2, 48, 144),
         ((20, 14), (1, 0), 6, 70, 140), ((14, 20), (0, 1), 6, 70, 140),
         ((40, 20), (1, 0), 2, 200, 400), ((40, 40), (1, 1), 2, 400, 800)]


def solve(n, per, levels, vc):
    c = context(n, per, 6, precision=0, mg_levels_max=levels, vc_visc=vc, vc_p=vc)
    cells = int(np.prod(c.dims(c.levels - 1)[0]))
    c.solve_viscous(2)
    c.solve_pressure(2)
    out = [c.get_field("ut", d) for d in range(c.dim)] + [c.get_field("p")]
    bytes_ = bfibm.footprint(c.prm)
    c.close()
    assert all(np.isfinite(a).all() for a in out)
    return out, bytes_, cells


@pytest.mark.parametrize("n,per,levels,rp,rv", CASES)
def test_matrix_is_its_sweeps(n, per, levels, rp, rv):
    want, plain, cells = solve(n, per, levels, 1)
    assert (rp, rv) == (cells, cells * len(n))
    for vc, limit in ((3, 384), (0, 800)):
        got, bytes_, _ = solve(n, per, levels, vc)
        rows = [r if r <= limit else 0 for r in (rp, rv)]
        assert bytes_ - plain == sum((8 * r * r + 255) // 256 * 256 for r in rows)
        for a, b in zip(got, want):
            assert np.abs(a - b).max() <= FP64_TOL * np.abs(b).max()
