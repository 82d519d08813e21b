"""The small-network fixpoint kernel against the host-driven queue of one-table
propagations (itself compared with the oracle in test_gpu_model.py): domains
and status after every cut, save and restore, on networks at the edges of the
kernel's rules (one table, more tables than descriptors kept in shared memory,
as many tables as it takes, rows per table at its limit and above it, few CTAs
so that misses are queued, no residues so that every value is scanned).
"""
import numpy as np
import pytest

from oracle import ct_oracle as O
from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


def _network(seed, nvars, ntables, arity, sizes, t):
    g = np.random.default_rng(seed)
    dom = [int(v) for v in g.choice(sizes, nvars)]
    spec = G.CspSpec(nvars=nvars, dom_lo=[0] * nvars, dom_size=dom)
    for _ in range(ntables):
        sc = [int(v) for v in g.choice(nvars, int(g.integers(arity[0], arity[1] + 1)), replace=False)]
        n = int(g.integers(t[0], t[1] + 1))
        spec.tables.append(G.TableSpec(sc, np.stack([g.integers(0, dom[v], n) for v in sc], axis=1).astype(np.int32)))
    return spec


def _model(spec, **opt):
    torch = torch_cuda()
    st, m = C.ct_model_create(spec.dom_lo, spec.dom_size, opt=C.make_options(**opt), stream=torch.cuda.current_stream())
    assert st == C.CT_OK
    for tb in spec.tables:
        assert C.ct_model_add_table(m, tb.scope, tb.tuples) >= 0, C.last_error()
    return m


@pytest.mark.parametrize("nvars,ntables,arity,sizes,t,opt", [
    (3, 1, (3, 3), [9], (60, 60), {}),
    (12, 65, (2, 4), [5, 33, 70], (200, 900), {}),
    (200, 512, (2, 3), [6, 40], (60, 150), {}),
    (1000, 512, (2, 4), [6, 40], (300, 900), {}),
    (16, 10, (8, 8), [128], (3000, 9000), {}),      # 1,024 rows per table
    (16, 10, (8, 8), [128, 129], (3000, 9000), {}),  # more in some: the general kernel
    (14, 9, (3, 5), [40], (2000, 9000), {"grid_blocks": 1}),
    (14, 9, (3, 5), [40], (2000, 9000), {"no_residues": 1}),
    (40, 6, (17, 32), [4, 7], (150, 400), {}),       # scopes beyond the descriptors' inline layout
])
def test_fixpoints_match_the_host_queue(nvars, ntables, arity, sizes, t, opt):
    spec = _network(nvars + ntables, nvars, ntables, arity, sizes, t)
    a, b = _model(spec, **opt), _model(spec, host_fixpoint=1)
    words = int(C.dom_layout(spec.dom_size)[0][-1])
    rng, level, ok, fails = G.Rng(nvars), 0, 0, 0
    sa, sb = C.ct_model_propagate(a), C.ct_model_propagate(b)
    assert sa == sb >= 0
    if sa != C.CT_OK:  # no solution at the root: nothing more to propagate
        assert C.ct_model_propagate(a) == C.ct_model_propagate(b) == C.CT_ERR_STATE
        C.ct_model_destroy(a)
        C.ct_model_destroy(b)
        return
    root = C.ct_model_get_domains(a, words)[1]
    assert np.array_equal(root, C.ct_model_get_domains(b, words)[1])
    masks = C.words_to_masks(root, spec.dom_size)
    for k in range(12):
        for m in (a, b):
            assert C.ct_model_save(m)[0] == C.CT_OK
        new = masks
        for _ in range(1 + k % 3):
            new, _ = (G.reset_step if rng.int(2) else G.delta_step)(rng, new)
        for m in (a, b):
            assert C.ct_model_set_domains(m, C.masks_to_words(new)) == C.CT_OK
        sa, sb = C.ct_model_propagate(a), C.ct_model_propagate(b)
        assert sa == sb >= 0, (k, C.last_error())
        level += 1
        if sa == C.CT_OK:
            ok += 1
            da = C.ct_model_get_domains(a, words)[1]
            assert np.array_equal(da, C.ct_model_get_domains(b, words)[1]), k
            masks = C.words_to_masks(da, spec.dom_size)
        if sa != C.CT_OK or k % 4 == 3:
            fails += sa != C.CT_OK
            back = rng.int(level)
            for m in (a, b):
                assert C.ct_model_restore(m, back) == C.CT_OK
            level = back
            da = C.ct_model_get_domains(a, words)[1]
            assert np.array_equal(da, C.ct_model_get_domains(b, words)[1]), k
            masks = C.words_to_masks(da, spec.dom_size)
    assert ok > 0
    C.ct_model_destroy(a)
    C.ct_model_destroy(b)


def test_search_equals_the_oracle_and_both_kernels_agree():
    spec = G.random_csp(77, 8, 6, 3, 5, 45)
    csp = O.Csp(spec.dom_lo, spec.dom_size)
    for tb in spec.tables:
        csp.add_table(tb.scope, tb.tuples)
    want = O.dfs(csp)
    for opt in ({}, {"grid_blocks": 2}, {"no_residues": 1}):
        m = _model(spec, **opt)
        st, got = C.ct_search_dfs(m, spec.nvars, 0, True)
        assert st == C.CT_OK, C.last_error()
        assert (got["nodes"], got["fails"], got["solutions"], got["max_depth"]) == \
            (want.nodes, want.fails, want.solutions, want.max_depth)
        C.ct_model_destroy(m)
