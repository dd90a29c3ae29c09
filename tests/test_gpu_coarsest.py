"""The coarsest level of FP64 contexts against the oracle: levels that only
just fit the cluster kernel's shared memory (csrc/cluster.cu), which
test_cluster_layout.py looks at on the CPU, and contexts whose coarsest level is
their only one, where each solve continues from the one before."""
import numpy as np
import pytest

from paper_1302_3663_gb300 import workloads as W

from helpers import assert_close, cell_mask, face_mask, pair, random_coefficients

pytestmark = pytest.mark.gpu

TOL = 1e-11   # a few V-cycles, as in test_gpu_stages.py


def contexts(n, per, seed, **kw):
    """A library and an oracle context with the same coefficients, iterates and
    right-hand sides; the pressure's has a mean, which the coarsest solve removes."""
    D, h = len(n), 1.0 / max(n)
    flow = max(a for a in range(D) if per[a])
    prm = W.base_params(D, n, per, flow, h, rho_ratio=2.0, mu_ratio=20.0, omega=2 * h,
                        omega_mu=2 * h, u_center=0.0, body_force=1.0, **kw)
    g, o = pair(dict(params=prm), load=False)
    rng = np.random.default_rng(seed)
    random_coefficients(g, o, rng, mu_ratio=20.0)
    for d in range(D):
        for which, scale in (("ut", 1.0), ("urhs", 1e2)):
            a = np.where(face_mask(g, d), scale * rng.normal(size=g.shape()), 0.0)
            g.set_field(which, a, d)
            o.set(which, a, d)
    for which, mean in (("p", 0.0), ("prhs", 0.25)):
        a = np.where(cell_mask(g), rng.normal(size=g.shape()) + mean, 0.0)
        g.set_field(which, a)
        o.set(which, a)
    return g, o


def solve_and_compare(g, o, cycles):
    assert g.solve_viscous(cycles) == cycles
    assert g.solve_pressure(cycles) == cycles
    o.solve_visc(cycles)
    o.solve_p(cycles)
    for d in range(g.dim):
        assert_close(g.get_field("ut", d), o.get("ut", d), TOL, "u~ %d" % d)
    assert_close(g.get_field("p"), o.get("p"), TOL, "p")


@pytest.mark.parametrize("n,per", [((100, 50, 100), (0, 0, 1)), ((90, 90, 64), (0, 0, 1)),
                                   ((604, 800), (1, 0))])
def test_coarsest_levels_at_the_edge_of_shared_memory(n, per):
    g, o = contexts(n, per, 21)
    solve_and_compare(g, o, 2)
    g.close()


# grids that cannot be halved (an odd half of a periodic axis), and one kept at one level; up to
# 800 unknowns a solve (a matrix's rows in deeper contexts) and more
ONE_LEVEL = [((22, 16), (1, 0), 6), ((14, 12), (1, 0), 6), ((6, 6, 6), (0, 0, 1), 6),
             ((7, 10, 4), (0, 0, 1), 6), ((8, 8, 16), (0, 0, 1), 1), ((32, 24), (1, 0), 1)]


@pytest.mark.parametrize("cycles", [3, 30])
@pytest.mark.parametrize("n,per,levels", ONE_LEVEL)
def test_one_level_continues_from_its_iterate(n, per, levels, cycles):
    g, o = contexts(n, per, 22, mg_levels_max=levels)
    assert g.levels == 1
    solve_and_compare(g, o, cycles)
    # the mean is taken off the right-hand side itself, which the residual reads
    assert_close(g.get_field("prhs"), o.get("prhs"), TOL, "prhs")
    g.close()


@pytest.mark.parametrize("n,per,levels", ONE_LEVEL)
def test_one_level_reaches_a_tolerance(n, per, levels):
    g, _ = contexts(n, per, 23, mg_levels_max=levels, vc_visc=0, vc_p=0, rtol=1e-6,
                    max_cycles=1000)
    for solve, which in ((g.solve_viscous, "res_visc"), (g.solve_pressure, "res_p")):
        assert 0 < solve(0) < 1000
        assert g.get_stats()[which] <= 1e-6
    g.close()
