"""currTable's non-zero word count against the words themselves, on both sides of
the size where a kernel counts them (24,576 words), at partial last words and
chunks, full, thinned and empty, with and without the words.
"""
import ctypes

import numpy as np
import pytest

from paper_2507_18413_gb300 import ct as C
from gpu_helpers import GpuTable, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t", [1, 33, 24_575 * 32, 24_575 * 32 + 1, 24_576 * 32 + 7, 1_000_003, 6_000_001])
def test_count_equals_the_words(t):
    torch_cuda()
    sizes = [64, 7]
    g = np.random.default_rng(t)
    tup = np.stack([g.integers(0, d, t) for d in sizes], axis=1).astype(np.int32)
    tup[: t // 3, 0] = np.arange(t // 3) * 64 // max(1, t)  # long runs without the kept values
    gt = GpuTable([0, 0], sizes, tup)
    full = [np.ones(d, bool) for d in sizes]
    for keep in (64, 40, 1):
        m = [f.copy() for f in full]
        m[0][: 64 - keep] = False
        st, _, _ = gt.propagate(m)
        if st != C.CT_OK:
            break
        w, nz = gt.currtable()
        valid = m[0][tup[:, 0]] & m[1][tup[:, 1]]
        pad = np.zeros(-t % 32, bool)
        expect = int(np.concatenate([valid, pad]).reshape(-1, 32).any(axis=1).sum())
        assert nz == int(np.count_nonzero(w)) == expect
        n = ctypes.c_int64(-1)
        assert C.load().ct_get_currtable(gt.h, None, ctypes.byref(n)) == C.CT_OK and n.value == expect
        assert C.load().ct_get_currtable(gt.h, None, None) == C.CT_OK
    gt.close()
