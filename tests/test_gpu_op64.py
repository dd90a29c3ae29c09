"""The FP64 operator passes of the mixed-precision solves (csrc/op64.cu; 2D:
csrc/mixed.cu) against the library's face-by-face FP64 residuals, which
test_gpu_stages.py compares with the oracle. Grids with ragged tiles and
chunks, more than one tile along x, periodic and walled axes in every place,
odd halves, one-level grids (the coarsest solve on the finest level) and grids
smaller than a tile."""
import numpy as np
import pytest

from paper_1302_3663_gb300 import bfibm, workloads as W

from helpers import cell_mask, face_mask

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
GRIDS = [((48, 20, 40), (0, 0, 1)), ((40, 22, 44), (1, 0, 1)), ((32, 36, 30), (1, 0, 0)),
         ((16, 18, 20), (1, 1, 1)), ((16, 20, 24), (1, 1, 1)), ((33, 13, 10), (0, 0, 1)),
         ((34, 14, 20), (0, 0, 1)), ((200, 6, 8), (0, 0, 1)), ((4, 4, 8), (0, 0, 1)),
         ((2, 2, 2), (1, 1, 1)), ((4, 4, 4), (1, 1, 1)), ((64, 32), (1, 0)), ((20, 14), (1, 0))]


def context(n, per, seed, **kw):
    D, h = len(n), 1.0 / max(n)
    flow = max(a for a in range(D) if per[a])
    prm = W.base_params(D, n, per, flow, h, rho_ratio=2.0, mu_ratio=50.0, omega=2 * h,
                        omega_mu=2 * h, u_center=0.0, body_force=1.0, **dict(dict(precision=1), **kw))
    c = bfibm.Context(prm)
    rng = np.random.default_rng(seed)
    sh = c.shape()
    for d in range(D):
        c.set_field("rho", rng.uniform(1, 2, sh), d)
    c.set_field("muc", 0.01 * np.exp(rng.uniform(0, np.log(50), sh)))
    for e in range(3 if D == 3 else 1):
        c.set_field("mue", 0.01 * np.exp(rng.uniform(0, np.log(50), sh)), e)
    c.build_coefficients()
    for d in range(D):
        m = face_mask(c, d)
        c.set_field("ut", np.where(m, rng.normal(size=sh), 0.0), d)
        c.set_field("urhs", np.where(m, 1e3 * rng.normal(size=sh), 0.0), d)
    m = cell_mask(c)
    b = np.where(m, 1e3 * rng.normal(size=sh), 0.0)
    c.set_field("prhs", np.where(m, b - b.sum() / m.sum(), 0.0))
    c.set_field("p", np.where(m, rng.normal(size=sh), 0.0))
    return c


@pytest.mark.parametrize("n,per", GRIDS)
def test_residuals_handed_to_fp32(n, per):
    c = context(n, per, 3)
    D, h = c.dim, c.prm["h"]
    c.solve_viscous(1)   # ends with the FP64 residual of its iterate as the FP32 right-hand side
    got = [c.get_field_f32("urhs", d) for d in range(D)]
    want = c.residual_viscous()
    u = max(np.abs(c.get_field("ut", d)).max() for d in range(D))
    f = max(np.abs(c.get_field("urhs", d)).max() for d in range(D))
    # every term of a face's residual is at most `big`; both sides round fewer than 64 of them
    big = f + u * (2.0 / c.prm["dt"] + 24 * 0.5 / h ** 2)
    for d in range(D):
        m = face_mask(c, d)
        err = np.abs(got[d].astype(float) - want[d])[m]
        assert (err <= 2.0 ** -24 * np.abs(want[d][m]) + 64 * EPS * big).all(), (d, err.max())
    c.solve_pressure(1)
    got, want, m = c.get_field_f32("prhs"), c.residual_pressure(), cell_mask(c)
    big = np.abs(c.get_field("prhs")).max() + 12 / h ** 2 * np.abs(c.get_field("p")).max()
    err = np.abs(got.astype(float) - want)[m]
    assert (err <= 2.0 ** -24 * np.abs(want[m]) + 64 * EPS * big).all(), err.max()
    st = c.get_stats()   # the reductions: the same residual's norm over |f|
    fn = np.linalg.norm(c.get_field("prhs")[m])
    assert abs(st["res_p"] * fn - np.linalg.norm(want[m])) <= 1e-10 * np.linalg.norm(want[m]) + \
        64 * EPS * big * np.sqrt(m.sum())
    c.close()


@pytest.mark.parametrize("n,per", GRIDS)
def test_flexible_cg_applies_the_same_operator(n, per):
    # the recurrence r -= alpha A p tracks the true residual only if w = A z is the operator
    # of the residual: at convergence the face-by-face residual agrees with the tolerance
    rtol = 1e-9
    c = context(n, per, 4, rtol=rtol, max_cycles=400, vc_visc=0, vc_p=0, krylov=1)
    cycles = c.solve_viscous(0)
    assert cycles < 400
    r = c.residual_viscous()
    rn = np.sqrt(sum((r[d][face_mask(c, d)] ** 2).sum() for d in range(c.dim)))
    fn = np.sqrt(sum((c.get_field("urhs", d)[face_mask(c, d)] ** 2).sum() for d in range(c.dim)))
    assert rn <= 2 * rtol * fn
    c.close()
