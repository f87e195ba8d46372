"""Contexts on threads of their own (a context is one thread's at a time, and
different ones run side by side): windows whose kernels need different amounts
of shared memory, made into integral images and classified at once.  No call
may fail, and each thread's results are those of the same steps alone."""

import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(6, 6), (10, 10), (24, 24), (32, 32)]


def _work(h, w, times, out):
    from paper_1306_1467_gb300 import vjb
    rng = np.random.default_rng(h * 100 + w)
    px = rng.integers(0, 256, (64, h, w), dtype=np.uint8)
    y = (np.arange(64) % 3 == 0).astype(np.uint8)
    stumps = [dict(feature=f, threshold=3, polarity=1, split=0, error=0.1, beta=0.1, alpha=1.0 + f) for f in range(5)]
    try:
        with vjb.Trainer(0) as prep, vjb.Trainer(0) as cls:
            prep.load_windows(px, y)
            cls.prepare(px, y)
            for _ in range(times):
                prep.build_integral()
                _, scores = cls.classify(px, stumps)
                out.append(np.concatenate([prep.get_integral().ravel(), scores]))
    except Exception as e:  # for the thread that compares
        out.append(e)


def test_window_sizes_side_by_side():
    alone, together = {}, {s: [] for s in SIZES}
    for s in SIZES:
        out = []
        _work(*s, 1, out)
        alone[s] = out[0]
    threads = [threading.Thread(target=_work, args=(*s, 400, together[s])) for s in SIZES]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for s in SIZES:
        for got in together[s]:
            if isinstance(got, Exception):
                raise got
            assert np.array_equal(got, alone[s]), s
        assert len(together[s]) == 400
