"""As many tables as the small-network kernel takes, over few variables, with a
solution planted: the root is feasible, fixpoints take several rounds and remove
values beyond the edit, levels and restores cross them (test_gpu_net.py's network
of these sizes is infeasible at its root, the second test's subject here). Against
the host-driven queue of one-table propagations.
"""
import numpy as np
import pytest

from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


def _network(seed, nvars, ntables, sizes, share):
    """Tables of `share` of their tuple space (at most 3,000 tuples), a solution among them."""
    g = np.random.default_rng(seed)
    dom = [int(v) for v in g.choice(sizes, nvars)]
    sol = [int(g.integers(0, d)) for d in dom]
    spec = G.CspSpec(nvars=nvars, dom_lo=[0] * nvars, dom_size=dom)
    for k in range(ntables):
        sc = [int(v) for v in g.choice(nvars, int(g.integers(2, 4)), replace=False)]
        ds = [dom[v] for v in sc]
        tup = G.distinct_uniform_tuples(seed + k, [0] * len(sc), ds, int(min(3000, max(2, share * np.prod(ds)))))
        if not (tup == [sol[v] for v in sc]).all(axis=1).any():
            tup[0] = [sol[v] for v in sc]
        spec.tables.append(G.TableSpec(sc, tup))
    return spec, sol


def _model(spec, **opt):
    torch = torch_cuda()
    st, m = C.ct_model_create(spec.dom_lo, spec.dom_size, opt=C.make_options(**opt), stream=torch.cuda.current_stream())
    assert st == C.CT_OK
    for tb in spec.tables:
        assert C.ct_model_add_table(m, tb.scope, tb.tuples) >= 0, C.last_error()
    return m


@pytest.mark.parametrize("nvars,opt", [(200, {}), (200, {"grid_blocks": 7}), (200, {"no_residues": 1})])
def test_512_tables_with_a_solution(nvars, opt):
    spec, sol = _network(nvars, nvars, 512, [6, 40], 0.4)
    a, b = _model(spec, **opt), _model(spec, host_fixpoint=1)
    words = int(C.dom_layout(spec.dom_size)[0][-1])
    assert C.ct_model_propagate(a) == C.ct_model_propagate(b) == C.CT_OK
    g, level, rounds, beyond, fails = np.random.default_rng(nvars), 0, 0, 0, 0
    for k in range(16):
        root = C.ct_model_get_domains(a, words)[1]
        assert np.array_equal(root, C.ct_model_get_domains(b, words)[1]), k
        masks = C.words_to_masks(root, spec.dom_size)
        for m in (a, b):
            assert C.ct_model_save(m) == (C.CT_OK, level)
        level += 1
        for v in g.choice(nvars, 6, replace=False):
            keep = g.random(spec.dom_size[v]) < 0.4
            if k % 5 != 4:
                keep[sol[v]] = True
            if (masks[v] & keep).any():
                masks[v] = masks[v] & keep
        edit = C.masks_to_words(masks)
        C.ct_model_reset_stats(a)
        for m in (a, b):
            assert C.ct_model_set_domains(m, edit) == C.CT_OK
        sa, sb = C.ct_model_propagate(a), C.ct_model_propagate(b)
        assert sa == sb >= 0, (k, C.last_error())
        if sa == C.CT_OK:
            da = C.ct_model_get_domains(a, words)[1]
            assert np.array_equal(da, C.ct_model_get_domains(b, words)[1]), k
            rounds = max(rounds, C.ct_model_get_stats(a)[1]["rounds"])
            beyond += not np.array_equal(da, edit)
        fails += sa != C.CT_OK
        if sa != C.CT_OK or k % 4 == 3:
            level = int(g.integers(0, level))
            for m in (a, b):
                assert C.ct_model_restore(m, level) == C.CT_OK
    assert rounds > 1 and beyond > 0
    C.ct_model_destroy(a)
    C.ct_model_destroy(b)


def test_an_infeasible_root_fails_on_both():
    spec, sol = _network(5, 200, 511, [6, 40], 0.4)
    v, w = spec.tables[0].scope[:2]
    # every tuple takes a value of v with one of w that another table forbids
    spec.tables.append(G.TableSpec([v, w], np.array([[sol[v], sol[w]]], np.int32)))
    spec.tables[0] = G.TableSpec([v, w], np.array([[(sol[v] + 1) % spec.dom_size[v], sol[w]]], np.int32))
    a, b = _model(spec), _model(spec, host_fixpoint=1)
    assert C.ct_model_propagate(a) == C.ct_model_propagate(b) == C.CT_INFEASIBLE
    assert C.ct_model_propagate(a) == C.ct_model_propagate(b) == C.CT_ERR_STATE
    C.ct_model_destroy(a)
    C.ct_model_destroy(b)
