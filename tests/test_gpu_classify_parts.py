"""The classifier's windows in parts: at 24 MiB a part, one part and a window
more, several with a ragged last one, and a call whose workspace is given back.
With more than one part the copies run on a stream of their own, which has to
come after the work already queued on the context's stream: windows in pinned
memory may still be on their way there.  Values are whole numbers and scores
FP64 sums in stump order, so the comparison is exact."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PART = 24 << 20


def _two_wide(px, f):
    """A feature of two rectangles side by side on every window, from pixel sums."""
    _, x, y, w, h = (int(v) for v in f)
    s = px[:, y: y + h, x: x + w].astype(np.int64)
    return s[:, :, w // 2:].sum((1, 2)) - s[:, :, : w // 2].sum((1, 2))


def _trainer(h, w, stream=None):
    from paper_1306_1467_gb300 import vjb
    tr = vjb.Trainer(0, stream=stream)
    rng = np.random.default_rng(h)
    feats = tr.prepare(rng.integers(0, 256, (4, h, w), dtype=np.uint8), np.array([0, 1, 0, 1], np.uint8))
    return tr, feats


def _expected(px, feats, T):
    rng = np.random.default_rng(T)
    two = np.flatnonzero((feats[:, 0] == 2) & (feats[:, 3] * feats[:, 4] <= 24))  # type 2H, small boxes
    stumps, score, half = [], np.zeros(px.shape[0]), 0.0
    for _ in range(T):
        f = int(rng.choice(two))
        v = _two_wide(px, feats[f])
        th, p, alpha = int(rng.integers(-40, 41)), int(rng.choice([-1, 1])), float(rng.exponential())
        stumps.append(dict(feature=f, threshold=th, polarity=p, split=0, error=0.1, beta=0.1, alpha=alpha))
        score = score + np.where(p * v < p * th, alpha, 0.0)
        half += alpha
    return stumps, score, (score >= 0.5 * half).astype(np.uint8)


def _part(h, w):
    return PART // (h * w) // 32 * 32


@pytest.mark.parametrize("h,w,n", [(24, 24, _part(24, 24)), (24, 24, _part(24, 24) + 1), (24, 24, 2 * _part(24, 24) + 33),
                                   (24, 24, 150_001), (32, 31, 4 * _part(32, 31) + 5), (4, 4, 2_000_000)])
def test_windows_in_parts(h, w, n):
    rng = np.random.default_rng(n)
    px = rng.integers(0, 256, (n, h, w), dtype=np.uint8)
    tr, feats = _trainer(h, w)
    with tr:
        stumps, score, label = _expected(px, feats, 5)
        for m in (n, n, n // 2, 3):  # a second call finds the first one's buffers, and smaller ones follow
            lab, sc = tr.classify(px[:m], stumps)
            assert np.array_equal(sc, score[:m])
            assert np.array_equal(lab, label[:m])


@pytest.mark.parametrize("n", [40_000, _part(24, 24) + 1000, 100_003])
def test_windows_still_being_written_on_the_stream(n):
    import torch
    px = np.random.default_rng(n).integers(0, 256, (n, 24, 24), dtype=np.uint8)
    on_device = torch.from_numpy(px).cuda()
    slow, fast = (torch.zeros(1 << 30, dtype=torch.uint8, device="cuda") for _ in range(2))
    pinned = torch.zeros((n, 24, 24), dtype=torch.uint8, pin_memory=True)
    stream = torch.cuda.Stream()
    tr, feats = _trainer(24, 24, stream.cuda_stream)
    with tr:
        stumps, score, label = _expected(px, feats, 5)
        tr.classify(px[: n // 2], stumps)  # the workspace and the copy stream are there
        for _ in range(3):
            pinned.zero_()
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                for _ in range(40):  # 10 ms and more before the download
                    slow.copy_(fast)
                pinned.copy_(on_device, non_blocking=True)
            lab, sc = tr.classify(pinned.numpy(), stumps)
            assert np.array_equal(sc, score)
            assert np.array_equal(lab, label)
