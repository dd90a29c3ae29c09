"""The pair sweep's packed lanes: rows of one parity side by side without gaps,
so that rows whose pairs are no multiple of 32 fill the warps and more rows fit
a block. Tile heights at the block's limit, odd and even row counts, rows of a
few pairs and of more than a hundred, against the ring sweep bit for bit."""
import numpy as np
import pytest

from test_gpu_pair import RING, sweep_with
from test_gpu_tma import context, random_inputs, sweep

pytestmark = pytest.mark.gpu

SHAPES = [((48, 40, 20), (18, 5)), ((48, 21, 12), (17, 4)), ((144, 12, 10), (5, 4)),
          ((72, 20, 18), (12, 3)), ((96, 17, 10), (8, 3)), ((160, 9, 8), (4, 3)),
          ((250, 6, 6), (2, 2)), ((4, 20, 8), (18, 3)), ((10, 30, 6), (14, 6))]

# blocks of 960 to 1024 threads, ragged last tiles
SHAPES += [((144, 30, 10), (12, 4)), ((160, 21, 8), (10, 3)), ((128, 28, 10), (14, 5)),
           ((250, 13, 6), (6, 3)), ((102, 40, 8), (18, 4))]


@pytest.mark.parametrize("n,pair", SHAPES)
def test_packed_rows_bit_identical_to_ring_sweep(n, pair):
    c = context(n, (0, 0, 1), 2)
    f = random_inputs(c, np.random.default_rng(3))
    shape = (pair[0], pair[1], 1, 0, 1)
    for x, y in zip(sweep_with(c, f, RING, 2), sweep_with(c, f, shape, 2)):
        assert np.isfinite(x).all() and np.array_equal(x, y)
    c.sweep_set_shape(0, 3, RING)
    a = sweep(c, f, 0, False, 2)
    c.sweep_set_shape(0, 3, shape)
    b = sweep(c, f, 0, False, 2)
    assert np.isfinite(a[0]).all() and np.array_equal(a[0], b[0])
    c.close()
