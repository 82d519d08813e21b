"""A network whose launches lie on both sides of the small-network kernel's line
(tables x segments of the first round): cuts of all variables and of one or two,
in turn, on the same tables, against the host-driven queue; the kernel that ran
shows in its plan phase, which the small-network kernel does not have.
"""
import numpy as np
import pytest

from paper_2507_18413_gb300 import ct as C
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


def _models(nv, ntables, d, t, sol, seed, opts):
    torch = torch_cuda()
    g = np.random.default_rng(seed)
    tabs = []
    for _ in range(ntables):
        sc = [int(v) for v in g.choice(nv, 3, replace=False)]
        tup = g.integers(0, d, (t, 3)).astype(np.int32)
        tup[0] = sol[sc]
        tabs.append((sc, tup))
    out = []
    for opt in opts:
        st, m = C.ct_model_create([0] * nv, [d] * nv, opt=C.make_options(**opt), stream=torch.cuda.current_stream())
        assert st == C.CT_OK
        for sc, tup in tabs:
            assert C.ct_model_add_table(m, sc, tup) == C.CT_OK, C.last_error()
        out.append(m)
    return out


@pytest.mark.parametrize("ntables,t,general", [
    (300, 49_000, True),    # 12 segments a table: 300 x 3,600, above the line
    (300, 45_000, False),   # 11: below it
    (20, 49_000, False),
])
def test_both_kernels_on_one_model(ntables, t, general):
    nv, d = 120, 128
    g = np.random.default_rng(ntables + t)
    sol = g.integers(0, d, nv)
    a, b = _models(nv, ntables, d, t, sol, 3, [{"profile": 1}, {"host_fixpoint": 1}])
    words = nv * 4
    assert C.ct_model_propagate(a) == C.ct_model_propagate(b) == C.CT_OK
    assert C.ct_model_get_stats(a)[1]["phase_seconds"][1] == 0  # (no table was cut yet)
    ran, rounds = [], 0
    level = 0
    for k in range(12):
        masks = C.words_to_masks(C.ct_model_get_domains(a, words)[1], [d] * nv)
        for m in (a, b):
            assert C.ct_model_save(m) == (C.CT_OK, level)
        level += 1
        heavy = k % 3 != 1
        for v in range(nv) if heavy else g.choice(nv, 2, replace=False):
            keep = g.random(d) < (0.5 if heavy else 0.3)
            keep[sol[v]] = True
            if k == 10:  # no solution: a variable keeps a single value at random
                keep[:] = False
                keep[int(g.integers(0, d))] = True
            masks[v] = masks[v] & keep
        if not all(m.any() for m in masks):
            masks = [m if m.any() else np.arange(d) == s for m, s in zip(masks, sol)]
        C.ct_model_reset_stats(a)
        for m in (a, b):
            assert C.ct_model_set_domains(m, C.masks_to_words(masks)) == C.CT_OK, C.last_error()
        sa, sb = C.ct_model_propagate(a), C.ct_model_propagate(b)
        assert sa == sb >= 0, (k, C.last_error())
        s = C.ct_model_get_stats(a)[1]
        ran.append((heavy, s["phase_seconds"][1] > 0))
        rounds = max(rounds, s["rounds"])
        if sa == C.CT_OK:
            assert np.array_equal(C.ct_model_get_domains(a, words)[1], C.ct_model_get_domains(b, words)[1]), k
        if sa != C.CT_OK or k % 4 == 3:
            back = int(g.integers(0, level))
            for m in (a, b):
                assert C.ct_model_restore(m, back) == C.CT_OK
            level = back
            assert np.array_equal(C.ct_model_get_domains(a, words)[1], C.ct_model_get_domains(b, words)[1]), k
    assert any(on for heavy, on in ran if heavy) == general, ran
    assert not any(on for heavy, on in ran if not heavy), ran
    assert rounds > 1
    for m in (a, b):
        C.ct_model_destroy(m)
