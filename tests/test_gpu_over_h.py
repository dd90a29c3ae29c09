"""Quotients by the mesh width (csrc/stencil.cu, over_h) against division: the projection
u = u~ - beta (p(F) - p(F-d)) / h with u~ = 0, beta = 1 and euler dt / sigma = 1 is that quotient
itself. Pressures over the whole range: ordinary, those whose quotients or their corrections
underflow, subnormal, zero, and those whose quotients overflow."""
import numpy as np
import pytest

from paper_1302_3663_gb300 import bfibm, workloads as W

from helpers import cell_mask, face_mask

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,per", [((16, 12, 20), (0, 0, 1)), ((64, 32), (1, 0))])
@pytest.mark.parametrize("h", [1.0 / 3.0, 0.1, 1.0 / 64.0, 0.7e-3, 1.9999999999999998, 37.3])
def test_gradients_round_as_a_division(n, per, h):
    D = len(n)
    flow = max(a for a in range(D) if per[a])
    c = bfibm.Context(W.base_params(D, n, per, flow, h, u_center=0.0, body_force=0.0, dt=1.0,
                                    omega=2 * h, omega_mu=2 * h))
    rng = np.random.default_rng(5)
    for d in range(D):
        c.set_field("ut", np.zeros(c.shape()), d)
        c.set_field("rho", np.ones(c.shape()), d)
    c.build_coefficients()
    for scale in (1.0, 1e-269, 1e-273, 1e-290, 1e-300, 1e-306, 1e-310, 1e-320, 0.0, 1e290, 8e307):
        p = np.where(cell_mask(c), scale * rng.uniform(-1, 1, c.shape()), 0.0)
        c.set_field("p", p)
        c.stage("project")
        for d in range(D):
            with np.errstate(over="ignore", under="ignore"):
                want = -(p - np.roll(p, 1, D - 1 - d)) / h
            m = face_mask(c, d)
            if per[d]:   # (the roll wraps over the stored extent, which is the cells there)
                assert c.shape()[D - 1 - d] == n[d]
            got = c.get_field("u", d)
            assert np.array_equal(got[m], want[m]), (scale, np.abs(got - want)[m].max())
    c.close()
