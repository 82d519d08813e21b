"""The ordering features against the float64 oracle on both of their paths:
networks of small tables (one kernel, a block per variable and table) and
networks with a table, a domain or a scope beyond its limits."""
import numpy as np
import pytest

from oracle import ct_oracle as O
from oracle import learned as L
from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,t", [
    ([5, 7, 9, 33, 64], [40, 129, 4_097]),
    ([40, 31, 20, 33], [32_768, 700]),      # 256 chunks: the most a block holds
    ([40, 31, 20, 33], [32_769, 700]),      # 257
    ([1_024, 12, 9], [9_000, 500]),         # 1,024 values
    ([1_025, 12, 9], [9_000, 500]),
])
def test_features_match_the_oracle(sizes, t):
    torch = torch_cuda()
    g = np.random.default_rng(sum(sizes) + sum(t))
    csp = O.Csp([0] * len(sizes), sizes)
    st, m = C.ct_model_create([0] * len(sizes), sizes, stream=torch.cuda.current_stream())
    assert st == C.CT_OK
    for n in t:
        sc = [int(v) for v in g.choice(len(sizes), 3, replace=False)]
        tup = np.stack([g.integers(0, sizes[v], n) for v in sc], axis=1).astype(np.int32)
        csp.add_table(sc, tup)
        assert C.ct_model_add_table(m, sc, tup) >= 0
    words = int(C.dom_layout(sizes)[0][-1])
    rng = G.Rng(len(t))
    assert C.ct_model_propagate(m) == C.CT_OK
    for k in range(4):
        masks = C.words_to_masks(C.ct_model_get_domains(m, words)[1], sizes)
        st, got = C.ct_model_features(m, len(sizes))
        assert st == C.CT_OK, C.last_error()
        want = L.features(csp, masks)
        assert np.all(np.abs(got - want) <= 1e-5 * np.maximum(1.0, np.abs(want))), k
        new, _ = (G.reset_step if k % 2 else G.delta_step)(rng, masks)
        assert C.ct_model_set_domains(m, C.masks_to_words(new)) == C.CT_OK
        if C.ct_model_propagate(m) != C.CT_OK:
            break
    C.ct_model_destroy(m)


@pytest.mark.parametrize("nvars", [1, 2, 7, 255, 257, 601])
def test_every_variable_is_published(nvars):
    """One variable to several per thread, most of them in no table; called again without a change."""
    torch = torch_cuda()
    sizes = [3 + v % 4 for v in range(nvars)]
    g = np.random.default_rng(nvars)
    csp = O.Csp([0] * nvars, sizes)
    st, m = C.ct_model_create([0] * nvars, sizes, stream=torch.cuda.current_stream())
    assert st == C.CT_OK
    for sc in {(0, nvars // 2, nvars - 1), (nvars - 1,)} if nvars > 2 else {(0,)}:
        tup = np.stack([g.integers(0, sizes[v], 50) for v in sc], axis=1).astype(np.int32)
        csp.add_table(list(sc), tup)
        assert C.ct_model_add_table(m, list(sc), tup) >= 0
    assert C.ct_model_propagate(m) == C.CT_OK
    masks = C.words_to_masks(C.ct_model_get_domains(m, int(C.dom_layout(sizes)[0][-1]))[1], sizes)
    want = L.features(csp, masks)
    for _ in range(3):
        st, got = C.ct_model_features(m, nvars)
        assert st == C.CT_OK, C.last_error()
        assert np.all(np.abs(got - want) <= 1e-5 * np.maximum(1.0, np.abs(want)))
    C.ct_model_destroy(m)
