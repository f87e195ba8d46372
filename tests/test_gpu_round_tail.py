"""The kernels after a plain round's search, at the edges of their split.

The cluster that ends a round re-scans lists of up to 16 features itself and
leaves longer ones to a second kernel; its blocks hold 256 samples each, two at
a time, sixteen to a pass.  Batched rounds take the same steps in kernels of
their own with the same sums in the same order, so stumps and weights must be
the same bits.  The initial weights, a cluster of 1,024 threads, are compared
with the oracle's: one FP32 rounding of a quotient formed in FP64.
"""

import numpy as np
import pytest

from oracle import oracle

pytestmark = pytest.mark.gpu

SIZES = [2, 3, 255, 256, 257, 512, 513, 8192, 8193, 16384, 16385, 24577, 32766]


def _windows(kind, n):
    rng = np.random.default_rng(n)
    y = np.zeros(n, np.uint8)
    y[rng.permutation(n)[: max(1, n // 3)]] = 1
    if kind == "single":  # hardly a tie
        return rng.integers(0, 256, (n, 7, 5), dtype=np.uint8), y
    if kind == "constant":  # every feature ties, and no round is kept
        return np.full((n, 5, 5), 9, np.uint8), y
    # equal rows in windows 2 wide: the features with two rectangles side by side tie at h (h + 1) / 2 heights
    # and places, those with three stacked at 3 (h = 5) or 4 + 1 (h = 6)
    h = {"fifteen": 5, "twenty_one": 6}[kind]
    return np.repeat(rng.integers(0, 256, (n, 1, 2), dtype=np.uint8), h, axis=1), y


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind", ["single", "fifteen", "twenty_one", "constant"])
def test_plain_rounds_equal_batched_ones(kind, n):
    from paper_1306_1467_gb300 import vjb
    px, y = _windows(kind, n)
    with vjb.Trainer(0) as tr:
        tr.prepare(px, y)
        _, plain = tr.train_strong(3)
        weights = tr.get_weights()
        listed = [d["candidates"] for d in tr.round_diag()]
    with vjb.Batch(vjb.Batch.table_bytes(n, *px.shape[1:])) as b:
        j = b.add_job(px, y, 3)
        b.train()
        batched = b.stumps(j)
        assert np.array_equal(b.get_weights(j), weights)
    assert plain == batched
    if n >= 255 and kind == "fifteen":
        assert max(listed) in (3, 15)
    if n >= 255 and kind == "twenty_one":
        assert max(listed) in (5, 21)


@pytest.mark.parametrize("n", [2, 3, 1023, 1024, 1025, 2049, 32766])
def test_initial_weights_match_oracle(n):
    from paper_1306_1467_gb300 import vjb
    px, y = _windows("fifteen", n)
    given = np.random.default_rng(n).random(n).astype(np.float32) + 0.5
    with vjb.Trainer(0) as tr:
        tr.prepare(px, y)
        np.testing.assert_allclose(tr.get_weights(), oracle.initial_weights(y), rtol=2.0**-24 * 1.001, atol=0)
        tr.set_weights(given)
        np.testing.assert_allclose(tr.get_weights(), oracle.normalize(given), rtol=2.0**-24 * 1.001, atol=0)
