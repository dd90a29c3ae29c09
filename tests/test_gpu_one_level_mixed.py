"""Mixed-precision contexts of a single level (odd extents, mg_levels_max = 1): the V-cycle is the
coarsest FP64 solve alone, on the level whose FP64 arrays hold the problem. Where the cluster kernel
holds it (csrc/cluster.cu) it converts in shared memory, whatever BFIBM_OPT_TAIL says; larger ones
run FP64 cycles."""
import numpy as np
import pytest

from paper_1302_3663_gb300 import bfibm

from helpers import cell_mask, face_mask
from test_gpu_op64 import context

pytestmark = pytest.mark.gpu

SMALL = [((33, 13, 10), (0, 0, 1), 6), ((16, 12, 20), (0, 0, 1), 1), ((22, 16), (1, 0), 6),
         ((6, 10, 6), (1, 0, 1), 6)]
LARGE = [((99, 75, 50), (0, 0, 1), 6), ((301, 400), (0, 1), 6), ((64, 48, 64), (1, 0, 1), 1)]


def fields(c):
    return [c.get_field("ut", d) for d in range(c.dim)] + [c.get_field("p")]


@pytest.mark.parametrize("krylov", [0, 1])
@pytest.mark.parametrize("n,per,levels", SMALL)
def test_solves_the_problem_it_was_given(n, per, levels, krylov):
    rtol, out = 1e-9, []
    for tail in (1 << 15, 0):
        c = context(n, per, 7, mg_levels_max=levels, rtol=rtol, max_cycles=4000, vc_visc=0, vc_p=0)
        assert c.levels == 1
        c.set_option(bfibm.OPT_TAIL, tail)
        c.set_option(bfibm.OPT_KRYLOV, krylov)
        rhs = [c.get_field("urhs", d) for d in range(c.dim)] + [c.get_field("prhs")]
        assert 0 < c.solve_viscous(0) < 4000 and 0 < c.solve_pressure(0) < 4000
        for a, b in zip(rhs, [c.get_field("urhs", d) for d in range(c.dim)] + [c.get_field("prhs")]):
            assert np.array_equal(a, b)
        rv, rp = c.residual_viscous(), c.residual_pressure()
        masks = [face_mask(c, d) for d in range(c.dim)]
        norm = lambda f: np.sqrt(sum((a[m] ** 2).sum() for a, m in zip(f, masks)))
        assert norm(rv) <= 2 * rtol * norm(rhs)   # (the CG's recurrence may end at twice rtol)
        m = cell_mask(c)
        assert np.linalg.norm(rp[m]) <= 2 * rtol * np.linalg.norm(rhs[-1][m])
        out.append(fields(c))
        c.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("call", ["solve", "step"])
@pytest.mark.parametrize("n,per,levels", LARGE)
def test_large_ones_are_the_fp64_cycles(n, per, levels, call):
    out = []
    for precision in (0, 1):
        c = context(n, per, 7, precision=precision, mg_levels_max=levels, vc_visc=2, vc_p=2)
        assert c.levels == 1
        if call == "step":
            rng = np.random.default_rng(8)
            for d in range(c.dim):
                c.set_velocity(d, np.where(face_mask(c, d), rng.normal(size=c.shape()), 0.0))
            c.step(1)
            out.append([c.get_velocity(d) for d in range(c.dim)] + [c.get_pressure()])
        else:
            c.solve_viscous(2)
            c.solve_pressure(2)
            out.append(fields(c))
        c.close()
    assert np.abs(out[0][-1]).max() > 0
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_a_persistent_batch_refuses_the_large_ones():
    b = bfibm.Batch(persistent=True, tune=False)
    cs = [context(n, per, 7, mg_levels_max=lv, vc_visc=0, vc_p=0, rtol=1e-6)
          for n, per, lv in (SMALL[0], LARGE[0])]
    b.add(cs[0])
    b.step()
    b.wait()
    b.add(cs[1])
    with pytest.raises(bfibm.BfibmError) as e:
        b.step()
    assert e.value.status == bfibm.EINVAL
    b.close()
    for c in cs:
        c.close()
