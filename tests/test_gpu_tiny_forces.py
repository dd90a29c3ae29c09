"""Spread forces far below one (csrc/lagrangian.cu): the fixed-point scale of the sums reaches the
top of the exponent range, where its reciprocal must stay a normal number."""
import numpy as np
import pytest

from helpers import face_mask, pair

from test_gpu_stages import ragged_duct

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1e-270, 1e-288, 1e-292, 1e-296, 1e-300, 1e-305])
def test_tiny_forces_spread_finitely(K):
    inst = ragged_duct()
    rng = np.random.default_rng(4)
    X = inst["X"] + rng.normal(scale=0.05 * inst["params"]["omega"], size=inst["X"].shape)
    for a in range(3):
        L = inst["params"]["n"][a] * inst["params"]["h"]
        X[:, a] = np.mod(X[:, a], L) if inst["params"]["periodic"][a] else np.clip(X[:, a], 0, L)
    g, o = pair(dict(inst, X=X, K=K * np.ones_like(inst["K"]), brk=np.full_like(inst["brk"], 5.0)))
    g.refresh()
    o.refresh()
    for d in range(3):
        a, b = g.get_field("force", d), o.get("force", d)
        m = face_mask(g, d)
        assert np.isfinite(a).all() and np.abs(b[m]).max() > 0
        # each node's share is rounded to a multiple of 1 / scale: 2^-1022 at the top of the
        # range, else 2^-59 of the bound on the sums, which is below 1e6 times the largest one;
        # node forces are rounded as well (springs' sums, subnormal below 2.2e-308 / 2^-53)
        tol = len(X) * max(2.0 ** -1022, 1e6 * 2.0 ** -59 * np.abs(b).max()) + 1e-300 * 2.0 ** -40
        assert np.abs(a - b)[m].max() <= tol, np.abs(a - b)[m].max()
    g.close()
