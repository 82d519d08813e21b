"""Networks whose tables lie at the edge of the miss search's rule (64 chunks: two
windows of every chunk; above: the live chunks): the fixpoint against the
host-driven queue, and the device search against the plain one, with one slot
and with more slots than open nodes.
"""
import numpy as np
import pytest

from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


def _model(sizes, tables, **opt):
    torch = torch_cuda()
    st, m = C.ct_model_create([0] * len(sizes), sizes, opt=C.make_options(**opt), stream=torch.cuda.current_stream())
    assert st == C.CT_OK
    for scope, tup in tables:
        assert C.ct_model_add_table(m, scope, tup) >= 0, C.last_error()
    return m


def _tables(t, seed):
    g = np.random.default_rng(seed)
    sizes = [14, 12, 33, 13, 11]
    out = []
    for scope in ([0, 1, 3, 4], [1, 2, 3], [0, 2, 4]):
        tup = np.unique(np.stack([g.integers(0, sizes[v], 3 * t) for v in scope], axis=1).astype(np.int32), axis=0)
        g.shuffle(tup)
        out.append((scope, np.ascontiguousarray(tup[:t])))
    return sizes, out


@pytest.mark.parametrize("t", [1, 128, 4_096, 4_097, 8_192, 8_193])
def test_fixpoints_at_the_window_rule(t):
    sizes, tables = _tables(t, t)
    a, b = _model(sizes, tables), _model(sizes, tables, host_fixpoint=1)
    words = int(C.dom_layout(sizes)[0][-1])
    sa, sb = C.ct_model_propagate(a), C.ct_model_propagate(b)
    assert sa == sb >= 0
    if sa == C.CT_OK:
        rng = G.Rng(t)
        masks = C.words_to_masks(C.ct_model_get_domains(a, words)[1], sizes)
        for k in range(10):
            for m in (a, b):
                assert C.ct_model_save(m)[0] == C.CT_OK
            new = (G.reset_step if k % 2 else G.delta_step)(rng, masks)[0]
            for m in (a, b):
                assert C.ct_model_set_domains(m, C.masks_to_words(new)) == C.CT_OK
            sa, sb = C.ct_model_propagate(a), C.ct_model_propagate(b)
            assert sa == sb >= 0
            if sa != C.CT_OK:
                break
            da = C.ct_model_get_domains(a, words)[1]
            assert np.array_equal(da, C.ct_model_get_domains(b, words)[1]), k
            masks = C.words_to_masks(da, sizes)
    C.ct_model_destroy(a)
    C.ct_model_destroy(b)


@pytest.mark.parametrize("t,slots,limit", [(400, 1, 0), (400, 64, 0), (1_500, 64, 0), (1_500, 64, 40)])
def test_device_search_counts_at_the_window_rule(t, slots, limit):
    sizes, tables = _tables(t, t + 1)
    a, b = _model(sizes, tables), _model(sizes, tables)
    st, d = C.ct_search_dfs(a, len(sizes), limit, True)
    assert st == C.CT_OK
    st, e, info = C.ct_search_batch_device(b, len(sizes), slots, 3, node_limit=limit)
    assert st == C.CT_OK
    if limit == 0:
        for key in ("nodes", "fails", "solutions"):
            assert d[key] == e[key], key
        assert np.array_equal(d["first_solution"], e["first_solution"])
    else:
        assert e["nodes"] == d["nodes"] == limit
    C.ct_model_destroy(a)
    C.ct_model_destroy(b)
