"""FP64 red-black sweeps by inverse diagonals (csrc/stencil.cu, k_v_rbgs, k_p_rbgs) against
division: the same numerator, and the quotient from an inverse in two parts (csrc/point.cuh,
pt_quot) is the rounded one except where it lies within about 2^-51 units in its last place of a
tie, which a few hundred thousand updates do not meet."""
import numpy as np
import pytest

from test_gpu_op64 import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,per", [((40, 22, 44), (1, 0, 1)), ((66, 6, 4), (0, 0, 1)),
                                   ((10, 14, 20), (0, 0, 1)), ((34, 6, 12), (0, 0, 1)),
                                   ((64, 32), (1, 0)), ((6, 132), (0, 1))])
def test_sweeps_round_as_a_division(n, per):
    # a mixed-precision context stores no inverse diagonals above its coarsest level and divides
    out = []
    for precision in (0, 1):
        c = context(n, per, 8, precision=precision)
        assert c.levels > 1
        c.smooth_viscous(0, 3)
        c.smooth_pressure(0, 3)
        out.append([c.get_field("ut", d) for d in range(c.dim)] + [c.get_field("p")])
        c.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b), np.abs(a - b).max()
