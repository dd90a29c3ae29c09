"""The FP32 sweeps' inverse viscous diagonals (csrc/mixed.cu, k_v_idg32): 1 / diagonal formed in
FP64 and rounded once to FP32, beside ties of that rounding and past FP32's range as well."""
import numpy as np
import pytest

from paper_1302_3663_gb300 import bfibm, workloads as W

from helpers import face_mask

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,per", [((16, 12, 20), (0, 0, 1)), ((64, 32), (1, 0))])
def test_inverse_diagonal_is_the_rounded_quotient(n, per):
    # without viscosity and with sigma / dt = 1 the diagonal is the density on the face
    D = len(n)
    flow = max(a for a in range(D) if per[a])
    c = bfibm.Context(W.base_params(D, n, per, flow, 1.0 / max(n), u_center=0.0, body_force=1.0,
                                    dt=1.0, precision=1))
    sh = c.shape()
    c.set_field("muc", np.zeros(sh))
    for e in range(3 if D == 3 else 1):
        c.set_field("mue", np.zeros(sh), e)
    rng = np.random.default_rng(3)
    rho = []
    for d in range(D):
        # 1 / rho within k 2^-49 of the middle of two FP32 neighbours
        f = rng.uniform(0.5, 2.0, sh).astype(np.float32)
        mid = f.astype(np.float64) + 0.5 * np.spacing(f).astype(np.float64)
        r = 1.0 / (mid * (1.0 + rng.integers(-8, 9, sh) * 2.0 ** -49))
        wide = rng.uniform(size=sh) < 0.2
        r = np.where(wide, 10.0 ** rng.uniform(-44, 44, sh), r)
        rho.append(r)
        c.set_field("rho", r, d)
    c.build_coefficients()
    for d in range(D):
        m = face_mask(c, d)
        with np.errstate(over="ignore", under="ignore"):
            want = (1.0 / rho[d]).astype(np.float32)
        assert np.array_equal(c.get_field_f32("idg", d)[m], want[m])
    c.close()
