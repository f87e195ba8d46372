"""Integral images and the strong classifier at the edges of their tiles: 32
windows a block, bands of rows of large windows, 128 stumps at a time, parts of
8 MiB of windows, and window sizes on both sides of what shared memory holds.
Integral images are whole numbers and scores FP64 sums in stump order, so the
comparison is exact."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _labels(n):
    return (np.arange(n) % 3 == 0).astype(np.uint8)


def _integral(px):
    n, h, w = px.shape
    ii = np.zeros((n, h + 1, w + 1), np.int32)
    ii[:, 1:, 1:] = px.astype(np.int64).cumsum(1).cumsum(2)
    return ii


@pytest.mark.parametrize("n,h,w", [(2, 1, 2), (31, 5, 7), (32, 10, 10), (33, 24, 24), (65, 9, 31), (40, 60, 60), (35, 3, 255),
                                   (33, 255, 2), (70, 100, 41)])
def test_integral_images(n, h, w):
    from paper_1306_1467_gb300 import vjb
    px = np.random.default_rng(n).integers(0, 256, (n, h, w), dtype=np.uint8)
    px[0] = 255
    with vjb.Trainer(0) as tr:
        tr.load_windows(px, _labels(n))
        tr.build_integral()
        assert np.array_equal(tr.get_integral(), _integral(px))


def _values(px, f):
    """One feature on every window, from pixel sums."""
    t, x, y, w, h = (int(v) for v in f)
    a, b = (w // 3, h) if t == 0 else (w, h // 3) if t == 1 else (w // 2, h) if t == 2 else (w, h // 2) if t == 3 else (w // 2, h // 2)

    def S(i, j):
        return px[:, y + j * b: y + (j + 1) * b, x + i * a: x + (i + 1) * a].astype(np.int64).sum((1, 2))
    if t == 0:
        return S(1, 0) - S(0, 0) - S(2, 0)
    if t == 1:
        return S(0, 1) - S(0, 0) - S(0, 2)
    if t == 2:
        return S(1, 0) - S(0, 0)
    if t == 3:
        return S(0, 1) - S(0, 0)
    return S(1, 0) + S(0, 1) - S(0, 0) - S(1, 1)


@pytest.mark.parametrize("n,h,w,T", [(1, 4, 4, 1), (31, 5, 7, 0), (32, 10, 10, 127), (33, 10, 11, 128), (200, 24, 24, 200),
                                     (1000, 9, 13, 129), (65, 20, 20, 700), (45, 41, 41, 30), (45, 60, 44, 30),
                                     (30011, 24, 24, 20), (8400, 32, 32, 9)])
def test_classifier(n, h, w, T):
    from paper_1306_1467_gb300 import vjb
    rng = np.random.default_rng(n + T)
    with vjb.Trainer(0) as tr:
        feats = tr.prepare(rng.integers(0, 256, (4, h, w), dtype=np.uint8), _labels(4))
        px = rng.integers(0, 256, (n, h, w), dtype=np.uint8)
        stumps, score, half = [], np.zeros(n), 0.0
        for _ in range(T):
            f = int(rng.integers(0, feats.shape[0]))
            v = _values(px, feats[f])
            th, p, alpha = int(rng.choice(v)) + int(rng.integers(0, 2)), int(rng.choice([-1, 1])), float(rng.exponential())
            stumps.append(dict(feature=f, threshold=th, polarity=p, split=0, error=0.1, beta=0.1, alpha=alpha))
            score = score + np.where(p * v < p * th, alpha, 0.0)
            half += alpha
        for _ in range(2):  # the second call finds the first one's buffers
            lab, sc = tr.classify(px, stumps)
            assert np.array_equal(sc, score)
            assert np.array_equal(lab, (score >= 0.5 * half).astype(np.uint8))
        few = min(n, 3)  # and a smaller one after it
        lab, sc = tr.classify(px[:few], stumps)
        assert np.array_equal(sc, score[:few])
