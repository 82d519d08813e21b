"""The ordering features on both sides of the line between their one-kernel path
and the two kernels: an entry's values times chunks, and a node's variables (the
oracle at the edges of the tables and domains is in test_gpu_features.py)."""
import numpy as np
import pytest

from oracle import ct_oracle as O
from oracle import learned as L
from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,ntables,t", [
    ([128, 12, 9, 40], 3, 30_000),    # 128 values x 256 chunks: the most an entry counts
    ([129, 12, 9, 40], 3, 30_000),    # 160 x 256
    ([512, 12, 9, 40], 3, 8_192),     # 512 x 64
    ([512, 12, 9, 40], 3, 8_193),     # 512 x 96
    ([20] * 256, 200, 1_500),         # a variable per thread
    ([20] * 257, 200, 1_500),
])
def test_features_match_the_oracle_at_the_line(sizes, ntables, t):
    torch = torch_cuda()
    nv = len(sizes)
    g = np.random.default_rng(nv + sizes[0] + t)
    csp = O.Csp([0] * nv, sizes)
    st, m = C.ct_model_create([0] * nv, sizes, stream=torch.cuda.current_stream())
    assert st == C.CT_OK
    sol = [int(g.integers(0, d)) for d in sizes]
    for k in range(ntables):
        sc = [0] + [int(v) for v in 1 + g.choice(nv - 1, 2, replace=False)] if k < 3 else \
            [int(v) for v in g.choice(nv, 3, replace=False)]
        tup = np.stack([g.integers(0, sizes[v], t) for v in sc], axis=1).astype(np.int32)
        tup[0] = [sol[v] for v in sc]
        csp.add_table(sc, tup)
        assert C.ct_model_add_table(m, sc, tup) >= 0
    words = int(C.dom_layout(sizes)[0][-1])
    for k in range(2):
        assert C.ct_model_propagate(m) == C.CT_OK
        masks = C.words_to_masks(C.ct_model_get_domains(m, words)[1], sizes)
        st, got = C.ct_model_features(m, nv)
        assert st == C.CT_OK, C.last_error()
        want = L.features(csp, masks)
        assert np.all(np.abs(got - want) <= 1e-5 * np.maximum(1.0, np.abs(want))), k
        # half of every domain's other values go, the solution stays
        for v in range(nv):
            keep = g.random(sizes[v]) < 0.5
            keep[sol[v]] = True
            masks[v] = masks[v] & keep
        assert C.ct_model_set_domains(m, C.masks_to_words(masks)) == C.CT_OK
    C.ct_model_destroy(m)


def test_a_policy_searches_alike_on_both_paths():
    """The first solution in depth-first order under a network's order: the plain
    search (one node at a time), and batches of few and of many entries."""
    torch = torch_cuda()
    nv, ntables, d, t = 100, 190, 8, 82
    g = np.random.default_rng(7)
    sol = [int(v) for v in g.integers(0, d, nv)]
    st, m = C.ct_model_create([0] * nv, [d] * nv, stream=torch.cuda.current_stream())
    assert st == C.CT_OK
    for k in range(ntables):
        sc = [int(v) for v in g.choice(nv, 3, replace=False)]
        tup = G.distinct_uniform_tuples(k, [0] * 3, [d] * 3, t)
        tup[0] = [sol[v] for v in sc]
        assert C.ct_model_add_table(m, sc, tup) >= 0
    st, net = C.ct_mlp_create(G.mlp_init_weights(3), stream=torch.cuda.current_stream())
    assert st == C.CT_OK
    assert C.ct_model_set_policy(m, net) == C.CT_OK
    st, want = C.ct_search_dfs(m, nv, 0, False)
    assert st == C.CT_OK and want["solutions"] == 1 and want["nodes"] > 1000
    for slots, split in ((8, 2), (64, 4)):
        st, got, _ = C.ct_search_batch(m, nv, slots, split, 0, False)
        assert st == C.CT_OK, C.last_error()
        assert got["first_solution"] == want["first_solution"], slots
    C.ct_model_destroy(m)
    C.ct_mlp_destroy(net)
