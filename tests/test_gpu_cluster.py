"""The cluster V-cycle (csrc/cluster.cu, BFIBM_OPT_TAIL) against a launch per
phase on grids where its slabs can go wrong: periodic and walled axes in every
place, odd coarse extents, rows of one or two points, fewer planes than CTAs,
2D, every level in the kernel. In mixed precision the bits agree; in FP64 the
launches round otherwise (divisions, the residual's form). The coarsest solve
as a matrix is compared with its sweeps."""
import numpy as np
import pytest

from paper_1302_3663_gb300 import bfibm

from test_gpu_op64 import context

pytestmark = pytest.mark.gpu

GRIDS = [((40, 22, 44), (1, 0, 1)), ((32, 36, 28), (1, 0, 0)), ((16, 20, 24), (1, 1, 1)),
         ((18, 18, 36), (0, 0, 1)), ((24, 12, 48), (0, 1, 1)), ((4, 20, 8), (0, 0, 1)),
         ((12, 12, 4), (0, 0, 1)), ((64, 32), (1, 0)), ((32, 48), (0, 1)), ((4, 8), (1, 1))]
# two V(2,2) cycles round each value some 4000 times (50 operations a sweep, 8 sweeps a level
# and cycle, 5 levels): 4000 x 2^-53 = 4.4e-13, with room for growth in between
FP64_TOL = 1e-11


def solve(n, per, tail, precision, **kw):
    c = context(n, per, 6, **dict(kw, precision=precision))
    c.set_option(bfibm.OPT_TAIL, tail)
    c.solve_viscous(2)
    c.solve_pressure(2)
    out = [c.get_field("ut", d) for d in range(c.dim)] + [c.get_field("p")]
    c.close()
    assert all(np.isfinite(a).all() for a in out)
    return out


@pytest.mark.parametrize("n,per", GRIDS)
def test_mixed_precision_bits(n, per):
    for a, b in zip(solve(n, per, 1 << 20, 1), solve(n, per, 0, 1)):
        assert np.array_equal(a, b), np.abs(a - b).max()


# the launches' FP32 residuals take two points along x: every pair beside a wall,
# planes of one and of several blocks, more cells than a cluster's slabs hold on the finest level
@pytest.mark.parametrize("n,per", [((4, 8, 8), (0, 0, 1)), ((12, 4, 12), (0, 1, 0)),
                                   ((4, 12, 8), (1, 0, 0)), ((68, 36, 20), (0, 0, 1)),
                                   ((44, 24, 72), (1, 1, 0))])
def test_residual_pairs_bits(n, per):
    for a, b in zip(solve(n, per, 1 << 15, 1), solve(n, per, 0, 1)):
        assert np.array_equal(a, b), np.abs(a - b).max()


@pytest.mark.parametrize("n,per", GRIDS)
def test_fp64_to_rounding(n, per):
    for a, b in zip(solve(n, per, 1 << 20, 0), solve(n, per, 0, 0)):
        assert np.abs(a - b).max() <= FP64_TOL * np.abs(b).max()


@pytest.mark.parametrize("n,per", GRIDS)
def test_coarsest_matrix_is_its_sweeps(n, per):
    # a context with one V-cycle per solve keeps the sweeps, more take the matrix
    for a, b in zip(solve(n, per, 1 << 20, 0, vc_visc=3, vc_p=3),
                    solve(n, per, 1 << 20, 0, vc_visc=1, vc_p=1)):
        assert np.abs(a - b).max() <= FP64_TOL * np.abs(b).max()


def test_coefficients_set_on_the_coarsest_level_are_used():
    # the inverse diagonals and the matrix follow a coefficient set by hand
    def run(scale):
        c = context((16, 16, 32), (0, 0, 1), 2, precision=0)
        l = c.levels - 1
        c.set_field("muc", scale * c.get_field("muc", 0, l), 0, l)
        c.solve_viscous(1)
        u = c.get_field("ut")
        c.close()
        return u
    assert np.array_equal(run(1.0), run(1.0))
    assert not np.array_equal(run(1.0), run(50.0))


@pytest.mark.parametrize("n,per", GRIDS + [((66, 6, 4), (0, 0, 1)), ((6, 130), (0, 1))])
def test_fp64_sweeps_with_inverse_diagonals(n, per):
    # an FP64 context multiplies by stored inverse diagonals, a mixed-precision one (whose finest
    # level stores none) divides: three sweeps of some 25 roundings each, diagonally dominant
    out = []
    for precision in (0, 1):
        c = context(n, per, 8, precision=precision)
        c.smooth_viscous(0, 3)
        c.smooth_pressure(0, 3)
        out.append([c.get_field("ut", d) for d in range(c.dim)] + [c.get_field("p")])
        c.close()
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 1e-13 * np.abs(b).max()
