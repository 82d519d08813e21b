"""A network's fixpoint whose bounded device waits run out (ct_model_arm_wait_timeout:
no barrier of the launch completes, every wait ends after a number of polls, the
kernel returns without publishing): the call returns CT_ERR_TIMEOUT, and as the
tables were left half-way, the model refuses every later propagation, restore
and search; the device and the stream stay usable.
"""
import numpy as np
import pytest

from oracle import ct_oracle as O
from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


def _model(spec, negative, **opt):
    torch = torch_cuda()
    st, m = C.ct_model_create(spec.dom_lo, spec.dom_size, opt=C.make_options(**opt), stream=torch.cuda.current_stream())
    assert st == C.CT_OK
    for k, tb in enumerate(spec.tables):
        assert C.ct_model_add_table(m, tb.scope, tb.tuples, negative=negative and k == 0) >= 0, C.last_error()
    return m


@pytest.mark.parametrize("negative", [False, True])  # the small-network kernel, the general one
def test_a_model_whose_wait_ran_out_refuses_later_calls(negative):
    spec = G.random_csp(77, 8, 6, 3, 5, 45)
    if negative:
        spec.tables[0].tuples = spec.tables[0].tuples[:20]
    m = _model(spec, negative)
    words = int(C.dom_layout(spec.dom_size)[0][-1])
    assert C.ct_model_arm_wait_timeout(m, 0) == C.CT_ERR_ARG
    assert C.ct_model_propagate(m) == C.CT_OK
    root = C.ct_model_get_domains(m, words)[1]
    assert C.ct_model_save(m) == (C.CT_OK, 0)
    masks = C.words_to_masks(root, spec.dom_size)
    new, _ = G.remove_random_values(G.Rng(4), masks, 2)
    assert C.ct_model_set_domains(m, C.masks_to_words(new)) == C.CT_OK
    assert C.ct_model_arm_wait_timeout(m, 2000) == C.CT_OK
    assert C.ct_model_propagate(m) == C.CT_ERR_TIMEOUT
    assert "wait ran out" in C.last_error()
    for _ in range(2):
        assert C.ct_model_propagate(m) == C.CT_ERR_TIMEOUT
        assert C.ct_model_restore(m, 0) == C.CT_ERR_TIMEOUT
    assert C.ct_search_dfs(m, spec.nvars, 0, True)[0] < 0
    assert C.ct_search_batch(m, spec.nvars, 4, 1)[0] < 0
    assert C.ct_model_destroy(m) == C.CT_OK
    # the device and the stream still work
    m = _model(spec, negative)
    assert C.ct_model_propagate(m) == C.CT_OK
    assert np.array_equal(C.ct_model_get_domains(m, words)[1], root)
    if not negative:
        csp = O.Csp(spec.dom_lo, spec.dom_size)
        for tb in spec.tables:
            csp.add_table(tb.scope, tb.tuples)
        want = O.dfs(csp)
        st, got = C.ct_search_dfs(m, spec.nvars, 0, True)
        assert st == C.CT_OK and (got["nodes"], got["solutions"]) == (want.nodes, want.solutions)
    C.ct_model_destroy(m)


def test_the_hook_is_for_one_launch_fixpoints():
    spec = G.random_csp(77, 8, 6, 3, 5, 45)
    m = _model(spec, False, host_fixpoint=1)
    assert C.ct_model_arm_wait_timeout(m, 100) == C.CT_ERR_ARG
    assert C.ct_model_propagate(m) == C.CT_OK
    C.ct_model_destroy(m)
