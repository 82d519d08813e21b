"""ct_call_stats.filter_bytes: the supports words filterDomains tests. A residue hit
costs 4 bytes, a window 512, and only a value that is scanned (or, in a negative
table, counted) over the whole index costs 16 bytes a live chunk: one that its
windows decide does not.
"""
import numpy as np
import pytest

from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G
from gpu_helpers import GpuTable

pytestmark = pytest.mark.gpu


def _calls(arity, d, t, n, negative=False, **opt):
    """Statistics of the successful calls with a value that neither residue nor window supports."""
    dom_lo, dom_size = [0] * arity, [d] * arity
    tup = G.distinct_uniform_tuples(5, dom_lo, dom_size, t)
    if negative:
        st, h = C.ct_create(arity, dom_lo, dom_size, tup, opt=C.make_options(**opt), negative=True)
        assert st == C.CT_OK, C.last_error()
    else:
        gt = GpuTable(dom_lo, dom_size, tup, opt=C.make_options(**opt))
        h = gt.h
    rng, masks, out = G.Rng(8), [np.ones(d, bool)] * arity, []
    C.ct_save(h)
    for k in range(n):
        new, _ = (G.reset_step if k % 2 else G.delta_step)(rng, masks)
        words = C.masks_to_words(new)
        st, _ = C.ct_propagate_host(h, words)
        s = C.ct_get_call_stats(h)[1]
        if st == C.CT_OK and s["hard"] > 0:
            out.append(s)
        masks = C.words_to_masks(words, dom_size)
        if st != C.CT_OK or k % 4 == 3:
            assert C.ct_restore(h, 0) == C.CT_OK
            C.ct_save(h)
            masks = [np.ones(d, bool)] * arity
    if negative:
        C.ct_destroy(h)
    else:
        gt.close()
    assert out, "no call had a hard value"
    return out


@pytest.mark.parametrize("arity,d,t,opt", [
    (3, 8, 200, {}),                      # one CTA
    (3, 8, 200, {"grid_blocks": 3}),      # the general kernel, windows that cover the table
    (3, 1500, 6000, {}),                  # a value per lane
])
def test_a_value_that_windows_decide_is_not_charged_a_scan(arity, d, t, opt):
    for s in _calls(arity, d, t, 24, **opt):
        assert s["filter_bytes"] == 4 * s["residue_hits"] + 512 * s["windows"], s


def test_scanned_values_are_charged_the_live_index():
    for s in _calls(3, 8, 200, 24, no_residues=1):
        assert s["filter_bytes"] == 16 * s["hard"] * s["live_chunks_out"] > 0, s


@pytest.mark.parametrize("opt", [{}, {"grid_blocks": 3}])
def test_counted_values_of_a_negative_table_are_charged_the_live_index(opt):
    for s in _calls(3, 5, 100, 24, negative=True, **opt):
        assert s["filter_bytes"] == 16 * s["hard"] * s["live_chunks_out"], s
