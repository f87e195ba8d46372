"""Contexts on threads of their own (a context is one thread's at a time, and
different ones run side by side): windows whose kernels need different amounts
of shared memory, made into integral images and classified at once.  No call
may fail, and each thread's results are those of the same steps alone."""

import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(6, 6), (10, 10), (24, 24), (32, 32)]


def _steps(h, w, times, out):
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
        _steps(*s, 1, out)
        alone[s] = out[0]
    threads = [threading.Thread(target=_steps, args=(*s, 400, together[s])) for s in SIZES]
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


def test_training_side_by_side():
    """Rounds whose lists go to the whole GPU (equal rows: every column pair of one
    height ties with the others), of four contexts at once."""
    from paper_1306_1467_gb300 import vjb

    def run(k, out):
        rng = np.random.default_rng(k)
        n, h = 3000 + 1111 * k, 8 + 6 * k
        y = (np.arange(n) % 3 == 0).astype(np.uint8)
        px = np.repeat((rng.integers(0, 200, (n, 1, 2)) + 20 * y[:, None, None] * np.array([0, 1])).astype(np.uint8), h, axis=1)
        try:
            with vjb.Trainer(0) as tr:
                tr.prepare(px, y)
                for _ in range(10):
                    tr.load_windows(px, y)
                    tr.build_integral()
                    tr.feature_count()
                    out.append((tr.train_strong(20), tr.get_weights().tobytes(), max(d["candidates"] for d in tr.round_diag())))
        except Exception as e:  # for the thread that compares
            out.append(e)

    alone, together = [], [[] for _ in range(4)]
    for k in range(4):
        out = []
        run(k, out)
        if isinstance(out[-1], Exception):
            raise out[-1]
        alone.append(out[0])
        assert out[0][2] > 16
    threads = [threading.Thread(target=run, args=(k, together[k])) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in range(4):
        assert together[k] == [alone[k]] * 10
