"""A stump count beyond the caller's array: the first stump that is none ends the
call, before anything of that count's size is made (24 bytes a stump)."""

import ctypes as C
import resource

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [2, 1000, 2**31 - 1])
def test_first_bad_stump_ends_the_call(T):
    from paper_1306_1467_gb300 import vjb
    px = np.random.default_rng(1).integers(0, 256, (8, 6, 6), dtype=np.uint8)
    with vjb.Trainer(0) as tr:
        tr.prepare(px, (np.arange(8) % 2).astype(np.uint8))
        stumps = (vjb.Stump * 2)()
        stumps[0].polarity, stumps[0].alpha = 1, 1.0  # stumps[1] has polarity 0
        lab = np.zeros(8, np.uint8)
        before = resource.getrusage(resource.RUSAGE_SELF).ru_maxrss
        rc = tr._lib.vjb_classify(tr._h, px.ctypes.data_as(C.c_void_p), 8, stumps, T, lab.ctypes.data_as(C.c_void_p), None)
        assert rc == vjb.EINVAL and b"stump 1 " in tr._lib.vjb_last_error()
        assert resource.getrusage(resource.RUSAGE_SELF).ru_maxrss - before < 1 << 20  # KiB: 1 GiB
        assert tr.classify(px, [stumps[0].as_dict()])[0].shape == (8,)  # the context goes on
