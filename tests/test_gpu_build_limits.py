"""Tables built where device memory is short (ct_debug_limit_bytes: a device of so
many bytes): the scratch that holds the tuples meanwhile is never what makes a
table fail. A table that fits by itself is built with the scratch cut down, put
aside for the table's buffers, or in host memory, and equals the oracle; one
byte less than the table needs is CT_ERR_OOM, every byte given back.
"""
import gc

import numpy as np
import pytest

from oracle import ct_oracle as O
from oracle import short as S
from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G
from gpu_helpers import GpuTable, compare_call, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture
def base():
    torch_cuda()
    C.load()
    gc.collect()  # tables of earlier tests left to the collector give their bytes back first
    yield C.ct_debug_device_bytes()[1]
    C.ct_debug_limit_bytes(-1)


def _inputs(kind):
    if kind == "short":
        dom_lo, dom_size = [0] * 4, [24] * 4
        return dom_lo, dom_size, G.short_tuples(4321, dom_lo, dom_size, 60_000, star_prob=0.1)
    dom_lo, dom_size, tup = G.large_table(77, 200_000)
    if kind == "dropped":  # every third tuple lies outside the domains
        tup = tup.copy()
        tup[::3, 2] = 40
    return dom_lo, dom_size, tup


@pytest.mark.parametrize("kind", ["whole", "dropped", "short"])
def test_a_table_that_fits_by_itself_is_built(base, kind):
    dom_lo, dom_size, tup = _inputs(kind)
    st, h = C.ct_create(len(dom_lo), dom_lo, dom_size, tup)
    assert st == C.CT_OK
    need = C.ct_debug_device_bytes()[1] - base
    C.ct_destroy(h)
    whole = tup.size * 4  # the whole list as scratch
    ones = [np.ones(d, bool) for d in dom_size]
    for spare in (0, 30_000, whole // 3, whole + 4096):
        C.ct_debug_limit_bytes(base + need + spare)
        gt = GpuTable(dom_lo, dom_size, tup)
        C.ct_debug_limit_bytes(-1)
        assert C.ct_debug_device_bytes()[1] == base + need
        if kind == "short":
            ret = S.retained_short(tup, dom_lo, dom_size)
            rng = G.Rng(3)
            for _ in range(3):
                new, _ = G.remove_random_values(rng, ones, 3)
                gt.save()
                st_o, out_o, _ = S.gac_table_short(ret, dom_lo, new)
                st_g, out_g, _ = gt.propagate(new)
                assert st_g == st_o == O.OK
                assert all(np.array_equal(a, b) for a, b in zip(out_g, out_o))
                gt.restore(0)
        else:
            ret = O.retained_tuples(tup, dom_lo, dom_size)
            assert compare_call(gt, ret, ones)[0] == O.OK
            new, _ = G.reset_step(G.Rng(3), ones)
            gt.save()
            compare_call(gt, ret, new)
        gt.close()
        gc.collect()
        assert C.ct_debug_device_bytes()[1] == base
    C.ct_debug_limit_bytes(base + need - 1)
    assert C.ct_create(len(dom_lo), dom_lo, dom_size, tup)[0] == C.CT_ERR_OOM
    assert C.ct_debug_device_bytes()[1] == base
