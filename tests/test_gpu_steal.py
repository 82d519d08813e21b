"""The device search with subtrees taken over between slots: counts, maximum
depth and the depth-first first solution equal the oracle's search (small
networks) and the plain search (larger ones), for few and many slots, shallow
splits (nearly every slot starts on a frame of another) and negative tables.
"""
import numpy as np
import pytest

from oracle import ct_oracle as O
from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu
KEYS = ("nodes", "fails", "solutions", "max_depth", "complete", "first_solution")


def _model(spec, negative=()):
    torch = torch_cuda()
    st, m = C.ct_model_create(spec.dom_lo, spec.dom_size, stream=torch.cuda.current_stream())
    assert st == C.CT_OK
    for k, tb in enumerate(spec.tables):
        assert C.ct_model_add_table(m, tb.scope, tb.tuples, negative=k in negative) >= 0, C.last_error()
    return m


@pytest.mark.parametrize("seed,nvars,ntables,d,t", [(1, 8, 5, 5, 60), (2, 9, 8, 4, 40), (3, 5, 2, 33, 400)])
@pytest.mark.parametrize("slots,split", [(2, 0), (33, 0), (96, 2)])
def test_small_networks_against_the_oracle(seed, nvars, ntables, d, t, slots, split):
    spec = G.random_csp(seed, nvars, ntables, 3, d, t)
    csp = O.Csp(spec.dom_lo, spec.dom_size)
    for tb in spec.tables:
        csp.add_table(tb.scope, tb.tuples)
    want = O.dfs(csp, count_all=True)
    m = _model(spec)
    for _ in range(2):  # (the second search reuses the slots and their buffers)
        st, got, info = C.ct_search_batch_device(m, spec.nvars, slots, split)
        assert st == C.CT_OK, C.last_error()
        assert (got["nodes"], got["fails"], got["solutions"], got["max_depth"]) == \
            (want.nodes, want.fails, want.solutions, want.max_depth)
        assert got["first_solution"] == (None if want.first_solution is None else list(want.first_solution))
        assert info["split_nodes"] + info["slot_nodes"] == got["nodes"]
    C.ct_model_destroy(m)


@pytest.mark.parametrize("seed,negative", [(0, ()), (5, (2, 5))])
def test_larger_networks_against_the_plain_search(seed, negative):
    spec = G.learned_csp(seed, nvars=(9, 9), dom=(8, 14), ntables=(13, 13), arity=(3, 4), tuples=(4e2, 5e3),
                         log2_solutions=-2.0)
    m = _model(spec, negative)
    st, want = C.ct_search_dfs(m, spec.nvars, 0, True)
    assert st == C.CT_OK
    steals = 0
    for slots, split in ((512, 1), (200, 8), (17, 4)):
        st, got, info = C.ct_search_batch_device(m, spec.nvars, slots, split)
        assert st == C.CT_OK, C.last_error()
        assert {k: got[k] for k in KEYS} == {k: want[k] for k in KEYS}
        steals += info["steals"]
    assert steals > 0
    C.ct_model_destroy(m)


def test_node_limit_ends_the_search():
    spec = G.learned_csp(3, nvars=(9, 9), dom=(8, 14), ntables=(13, 13), arity=(3, 4), tuples=(4e2, 5e3),
                         log2_solutions=0.0)
    m = _model(spec)
    for limit in (1, 40, 700):
        st, got, _ = C.ct_search_batch_device(m, spec.nvars, 64, 2, limit)
        assert st == C.CT_OK, C.last_error()
        assert got["nodes"] == limit and not got["complete"]
    C.ct_model_destroy(m)
