"""The allocation-free screen at the edges of its stages (16 lines of 64
entries, half a line a lane) against FP64 minima of the same table."""

import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# one lane, part of a stage, whole stages, one line more, the index limit
SIZES = [(1, 64), (2, 64), (33, 64), (64, 64), (65, 128), (511, 512), (960, 960), (961, 1024), (1024, 1024), (1025, 1088),
         (2048, 2112), (3000, 3008), (15000, 15040), (32766, 32768)]


@pytest.mark.parametrize("n,npad", SIZES)
@pytest.mark.parametrize("ctas", [0, 1, 1024])
def test_errors_at_stage_edges(n, npad, ctas):
    import torch
    from paper_1306_1467_gb300 import vjb
    lib = vjb.load_library()
    rng = np.random.default_rng(n)
    F = 37
    order = np.stack([rng.permutation(n) for _ in range(F)])
    flag = rng.random((F, n)) < rng.random((F, 1))
    flag[:, -1] = True
    rows = np.full((F, npad), n, np.uint16)
    rows[:, :n] = order | (flag.astype(np.uint16) << 15)
    rows[:, n:] += rng.integers(0, 32768 - n, (F, npad - n)).astype(np.uint16)  # any index from n on is padding
    w = np.exp(rng.uniform(-3, 3, n)).astype(np.float32)
    w /= w.astype(np.float64).sum()
    y = rng.random(n) < 0.4
    v = np.append(np.where(y, w, -w), 0).astype(np.float32)
    tp, tn = float(w[y].astype(np.float64).sum()), float(w[~y].astype(np.float64).sum())
    D = np.cumsum(v[:-1].astype(np.float64)[order], axis=1)
    want = np.minimum(tp - np.maximum(np.where(flag, D, -np.inf).max(1), 0), tn + np.minimum(np.where(flag, D, np.inf).min(1), 0))
    dev = [torch.from_numpy(a).cuda() for a in (rows.view(np.int16), v)]
    err, best, at = torch.full((F,), -1.0).cuda(), torch.zeros(1).cuda(), torch.zeros(1, dtype=torch.int32).cuda()
    p = [ctypes.c_void_p(t.data_ptr()) for t in (*dev, err, best, at)]
    rc = lib.vjb_screen_noalloc(p[0], p[1], n, npad, F, tp, tn, ctas, p[2], p[3], p[4], None)
    assert rc == vjb.OK, lib.vjb_last_error()
    torch.cuda.synchronize()
    got = err.cpu().numpy().astype(np.float64)
    # the screening bound: 35 u of the weight total, and the class totals' rounding
    assert np.max(np.abs(got - want)) <= 36 * 2.0 ** -24
    assert best.item() == err.min().item() and at.item() == int(err.argmin().item())
