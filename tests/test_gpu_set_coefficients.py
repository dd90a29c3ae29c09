"""Coefficients set by hand: each set costs its copy, whatever is formed from them (inverse
diagonals, the coarsest solve's matrices) is formed once, before the next sweep or cycle, and
follows every one of them."""
import time

import numpy as np
import pytest

from paper_1302_3663_gb300 import bfibm

from test_gpu_op64 import context

pytestmark = pytest.mark.gpu


def coefficients(c, level):
    return ([("beta", d) for d in range(c.dim)] + [("m", d) for d in range(c.dim)] + [("muc", 0)] +
            [("mue", e) for e in range(3 if c.dim == 3 else 1)])


@pytest.mark.parametrize("precision", [0, 1])
def test_a_set_costs_its_copy(precision):
    import torch
    c = context((64, 64, 128), (0, 0, 1), 4, precision=precision)
    for level in (0, c.levels - 1):
        t = torch.ones(c.shape(level), dtype=torch.float64, device="cuda")

        def best(name, comp):
            b = 1e9
            for _ in range(30):
                t0 = time.perf_counter()
                c.set_field_dev(name, t.data_ptr(), comp, level)
                b = min(b, time.perf_counter() - t0)
            return b
        plain = best("ut", 0)
        # the same bytes by the same copy; the diagonals alone would take several times as long
        for name, comp in coefficients(c, level):
            assert best(name, comp) <= 2.0 * plain, (name, level)
    c.close()


@pytest.mark.parametrize("n,per", [((16, 16, 32), (0, 0, 1)), ((32, 16), (1, 0))])
def test_sweeps_follow_every_coefficient(n, per):
    # against a mixed-precision context, which divides by the diagonal on its finest level; each
    # field changes after the inverses have been used
    cs = [context(n, per, 6, precision=p) for p in (0, 1)]
    for name, comp in coefficients(cs[0], 0):
        out = []
        for c in cs:
            c.set_field(name, 1.7 * c.get_field(name, comp), comp)
            c.smooth_viscous(0, 1)
            c.smooth_pressure(0, 1)
            out.append([c.get_field("ut", d) for d in range(c.dim)] + [c.get_field("p")])
        for a, b in zip(*out):
            assert np.array_equal(a, b), (name, comp, np.abs(a - b).max())
    for c in cs:
        c.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("call", ["solve", "step"])
def test_cycles_follow_the_coarsest_coefficients(precision, call):
    # set after or before the first use of the inverses: the same; not set: another result
    def run(when):
        c = context((16, 16, 32), (0, 0, 1), 6, precision=precision)
        c.refresh()
        l = c.levels - 1

        def change():
            for name, comp in coefficients(c, l):
                c.set_field(name, 3.0 * c.get_field(name, comp, l), comp, l)
        if when == "before":
            change()
        c.smooth_pressure(l, 1)   # uses the coarsest inverses
        if when == "after":
            change()
        if call == "step":
            c.step(1)
            out = [c.get_velocity(d) for d in range(c.dim)] + [c.get_pressure()]
        else:
            c.solve_viscous(3)
            c.solve_pressure(3)
            out = [c.get_field("ut", d) for d in range(c.dim)] + [c.get_field("p")]
        c.close()
        return out
    after, before, never = run("after"), run("before"), run("never")
    assert all(np.array_equal(a, b) for a, b in zip(after, before))
    assert any(not np.array_equal(a, b) for a, b in zip(after, never))


def test_a_new_batch_plan_follows_them():
    # the plan's capture queues the coefficients' build without running it: what was set by hand
    # before the first batch step counts in that step
    def run(change):
        c = context((16, 16, 32), (0, 0, 1), 6, precision=1, vc_visc=0, vc_p=0, rtol=1e-6)
        c.refresh()
        l = c.levels - 1
        if change:
            for name, comp in coefficients(c, l):
                c.set_field(name, 3.0 * c.get_field(name, comp, l), comp, l)
        b = bfibm.Batch(persistent=True, tune=False)
        if change == "formed":
            c.smooth_pressure(l, 0)
        b.add(c)
        b.step()
        b.wait()
        out = [c.get_velocity(d) for d in range(c.dim)] + [c.get_pressure()]
        b.close()
        c.close()
        return out
    late, formed, never = run("late"), run("formed"), run("")
    assert all(np.array_equal(a, b) for a, b in zip(late, formed))
    assert any(not np.array_equal(a, b) for a, b in zip(late, never))
