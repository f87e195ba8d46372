"""The sorted table where a thread block's share of a row changes, through the C ABI.

Feature values are read eight windows at a time, and the packed sort's blocks
hold 128 to 512 threads of 8 to 64 items: the last and first sample counts of
each block shape, and every remainder of eight windows.  Every row must be the
samples in value order, ties by index, with the split flags.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EDGES = [3584, 3585, 6144, 6145, 9216, 9217, 11264, 11265, 12288, 13312, 13313, 16896, 16897, 18432, 18433, 20736, 20737]
REMAINDERS = [n + r for n in (32, 4720, 15000) for r in range(8)]


@pytest.mark.parametrize("n", EDGES + REMAINDERS)
def test_rows_at_block_shape_edges(n):
    from paper_1306_1467_gb300 import vjb
    rng = np.random.default_rng(n)
    px = rng.integers(0, 256, (n, 5, 4), dtype=np.uint8)
    with vjb.Trainer(0) as tr:
        F = tr.prepare(px, (np.arange(n) % 3 == 0).astype(np.uint8)).shape[0]
        got, vals = tr.sorted_rows(0, F), tr.feature_values(0, F)
    order = np.argsort(vals, axis=1, kind="stable")
    assert np.array_equal(got & 0x7FFF, order)
    v = np.take_along_axis(vals, order, axis=1)
    flag = np.ones(v.shape, bool)
    flag[:, :-1] = v[:, :-1] < v[:, 1:]
    assert np.array_equal((got >> 15).astype(bool), flag)
