"""Rounds by the length of their list: of a run a warp, of two runs a warp (above
8), the longest that the cluster keeps (16), the shortest that goes to the
whole GPU (17), one with a feature for every block, and several for each.

Windows of grey columns, with faces and non-faces told apart (but for a share of
them) by the step from one column to the next in the top `a` rows, zeros below.
Every feature whose value is a multiple of that step ties, and no other comes
near: a list's length is the number of those features, counted here from their
values.  Batched rounds take the same steps in kernels of their own, with the same
sums in the same order, so stumps, weights and outcomes are the same bits.
"""

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


def _windows(n, h, w, a, wrong):
    rng = np.random.default_rng(n + h)
    y = np.zeros(n, np.uint8)
    y[rng.permutation(n)[: max(1, n // 3)]] = 1
    left = rng.integers(60, 196, n)
    step = np.where(rng.random(n) < wrong, -1, 1) * np.where(y == 1, 1, -1) * rng.integers(1, 60, n)
    px = np.zeros((n, h, w), np.uint8)
    px[:, :a, 0] = left[:, None]
    px[:, :a, 1] = (left + step)[:, None]
    return px, y


def _ties(h, w, a):
    one = np.zeros((2, h, w), np.uint8)
    one[0, :a, 0] = one[1, :a, 1] = 1
    left, right = O.feature_values_direct(one, O.haar_enumerate(w, h)[0]).T
    return int(((left == -right) & (left != 0)).sum())


SHAPES = [(3, 2, 1, 4), (6, 2, 1, 9), (5, 2, 4, 16), (7, 3, 1, 17), (24, 2, 24, 300), (40, 2, 5, 278), (100, 2, 100, 5050)]


@pytest.mark.parametrize("h,w,a,listed", SHAPES)
@pytest.mark.parametrize("n,wrong", [(257, 0.2), (2500, 0.2), (8193, 0.2), (32766, 0.2), (300, 0.0), (16385, 0.0)])
def test_lists(n, wrong, h, w, a, listed):
    from paper_1306_1467_gb300 import vjb
    assert _ties(h, w, a) == listed
    px, y = _windows(n, h, w, a, wrong)
    with vjb.Trainer(0) as tr:
        tr.prepare(px, y)
        status, plain = tr.train_strong(3)
        weights = tr.get_weights()
        assert tr.round_diag()[0]["candidates"] == listed
    with vjb.Batch(vjb.Batch.table_bytes(n, h, w)) as b:
        j = b.add_job(px, y, 3)
        b.train()
        assert b.job_state(j) == (len(plain), status)
        assert plain == b.stumps(j)
        assert np.array_equal(b.get_weights(j), weights)
    if wrong:
        assert len(plain) >= 1 and 0.0 < plain[0]["error"] < 0.5
    else:
        assert status == vjb.DONE_PERFECT and len(plain) == 1 and plain[0]["error"] == 0.0


@pytest.mark.parametrize("n", [256, 5000, 32766])
def test_no_feature_better_than_chance(n):
    from paper_1306_1467_gb300 import vjb
    px = np.full((n, 5, 5), 9, np.uint8)  # every feature ties, and no round is kept
    y = (np.arange(n) % 2).astype(np.uint8)
    with vjb.Trainer(0) as tr:
        tr.prepare(px, y)
        w0 = tr.get_weights()
        assert tr.train_strong(3) == (vjb.DONE_NOGAIN, [])
        assert np.array_equal(tr.get_weights(), w0)
        assert tr.info()["candidates"] == tr.info()["features"]
    with vjb.Batch(vjb.Batch.table_bytes(n, 5, 5)) as b:
        j = b.add_job(px, y, 3)
        b.train()
        assert b.job_state(j) == (0, vjb.DONE_NOGAIN)


def test_a_list_for_the_whole_gpu_costs_little_more():
    """What follows the search at 32,766 samples: 37 us with 4 features listed and
    57 with 17 or a few more; 403 when one block updated all the weights."""
    from paper_1306_1467_gb300 import vjb

    def after_search(h, w, a):
        px, y = _windows(32766, h, w, a, 0.2)
        times = []
        with vjb.Trainer(0) as tr:
            tr.prepare(px, y)
            w0 = tr.get_weights()
            for _ in range(15):
                tr.set_weights(w0)
                tr.set_timing(True)
                tr.train_strong(1)
                t = tr.timing()
                times.append(t["round_ms_total"] - t["search_ms_total"])
        return float(np.median(times[3:]))

    assert after_search(7, 3, 1) < 4 * after_search(3, 2, 1)


@pytest.mark.parametrize("h,w,a", [(25, 28, 1), (32, 32, 2), (40, 37, 3)])
def test_lists_of_large_windows(h, w, a):
    """More features than the tail asks for at once (196,608), ties among the last ones."""
    from paper_1306_1467_gb300 import vjb
    px, y = _windows(257, h, w, a, 0.2)
    with vjb.Trainer(0) as tr:
        tr.prepare(px, y)
        _, plain = tr.train_strong(2)
        weights = tr.get_weights()
        assert tr.round_diag()[0]["candidates"] == _ties(h, w, a)
    with vjb.Batch(vjb.Batch.table_bytes(257, h, w)) as b:
        j = b.add_job(px, y, 2)
        b.train()
        assert plain == b.stumps(j) and np.array_equal(b.get_weights(j), weights)


def test_large_windows_cost_little_more():
    """What follows the search with one feature listed, 300 samples: 25 us at 24x24
    and 35 at 48x48 (2,570,880 errors to look through); 65 with a load at a time."""
    from paper_1306_1467_gb300 import vjb

    def after_search(side):
        px = np.random.default_rng(side).integers(0, 256, (300, side, side), dtype=np.uint8)
        with vjb.Trainer(0) as tr:
            tr.load_windows(px, (np.arange(300) % 3 == 0).astype(np.uint8))
            tr.build_integral()
            tr.feature_count()
            tr.train_strong(3)
            times = []
            for _ in range(15):
                tr.set_timing(True)
                tr.train_strong(4)
                t = tr.timing()
                times.append(t["round_ms_total"] - t["search_ms_total"])
        return float(np.median(times))

    assert after_search(48) < 1.8 * after_search(24)
