"""The sorted table at the edges of every sort variant, through the C ABI.

The packed sort has a variant per range of sample counts (threads per CTA times
items per thread), takes one to three digit passes by the span of a feature's
values, evaluates small boxes from 16-bit integral images two windows to a
word, and leaves rows whose span and sample index exceed 32 bits to a second
sort.  Every row must be the samples in value order, ties by index, with the
split flags; whole numbers, so the comparison is exact.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# the last and the first sample count of each variant, remainders of 4, 32 and
# 256 samples, and the limits of the two weight copies
SIZES = [2, 3, 5, 31, 33, 255, 257, 1021, 1024, 1025, 2048, 2049, 3072, 3073, 4096, 4097, 5120, 5121, 6146, 7168, 7171,
         8192, 8193, 10240, 10241, 12289, 14336, 14339, 15360, 15361, 16351, 16352, 16384, 16385, 17920, 17921, 19200,
         19201, 20480, 20481, 24576, 24577, 28672, 28673, 32766]


def _check(px, y, picks=None):
    from paper_1306_1467_gb300 import vjb
    with vjb.Trainer(0) as tr:
        F = tr.prepare(px, y).shape[0]
        for f0 in range(0, F, 64) if picks is None else picks:
            nf = min(64, F - int(f0))
            got = tr.sorted_rows(int(f0), nf)
            vals = tr.feature_values(int(f0), nf)
            order = np.argsort(vals, axis=1, kind="stable")
            assert np.array_equal(got & 0x7FFF, order), f0
            v = np.take_along_axis(vals, order, axis=1)
            flag = np.ones(v.shape, bool)
            flag[:, :-1] = v[:, :-1] < v[:, 1:]
            assert np.array_equal((got >> 15).astype(bool), flag), f0


def _labels(n):
    return (np.arange(n) % 3 == 0).astype(np.uint8)


@pytest.mark.parametrize("n", SIZES)
def test_rows_at_variant_edges(n):
    rng = np.random.default_rng(n)
    _check(rng.integers(0, 256, (n, 4, 5), dtype=np.uint8), _labels(n))


@pytest.mark.parametrize("n", [600, 4096, 15000, 18300, 32766])
@pytest.mark.parametrize("kind", ["two_values", "mostly_one", "constant", "extremes"])
def test_rows_with_many_ties(n, kind):
    rng = np.random.default_rng(n + 1)
    if kind == "two_values":
        px = rng.integers(0, 2, (n, 4, 5), dtype=np.uint8) * 255
    elif kind == "mostly_one":
        px = np.where(rng.random((n, 4, 5)) < 0.02, rng.integers(0, 256, (n, 4, 5)), 7).astype(np.uint8)
    elif kind == "constant":
        px = np.full((n, 4, 5), 200, np.uint8)
    else:  # boxes at both ends of their value range
        px = np.repeat(rng.integers(0, 2, (n, 1, 5), dtype=np.uint8) * 255, 4, axis=1)
    _check(px, _labels(n))


@pytest.mark.parametrize("n,h,w", [(700, 40, 41), (4100, 33, 30), (16500, 48, 12), (900, 17, 16)])
def test_rows_of_large_boxes(n, h, w):
    """Boxes above 257 pixels (32-bit integral images), three digit passes and rows listed for the second sort."""
    rng = np.random.default_rng(h)
    px = np.where(rng.random((n, 1, 1)) < 0.5, rng.integers(0, 256, (n, h, w)), rng.integers(0, 2, (n, h, 1)) * 255)
    from paper_1306_1467_gb300 import vjb
    px = px.astype(np.uint8)
    with vjb.Trainer(0) as tr:
        F = tr.prepare(px[:4], _labels(4)).shape[0]
    _check(px, _labels(n), picks=sorted(rng.integers(0, F - 64, 6)) + [F - 64])
