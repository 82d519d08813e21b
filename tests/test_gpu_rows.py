"""Calls of exactly n rows, n at the edges of the update's batches and of their
groups (4, 8 and 16 rows), of one variable and of two, on a table of the
one-CTA kernel, of the general kernel and in a network of one table; every
result compared with the oracle.
"""
import numpy as np
import pytest

from oracle import ct_oracle as O
from paper_2507_18413_gb300 import ct as C
from gpu_helpers import GpuTable, compare_call, torch_cuda

pytestmark = pytest.mark.gpu

ROWS = [1, 3, 4, 5, 7, 8, 9, 12, 13, 15, 16, 17, 20, 33]


def _cuts(sizes, n):
    """Masks whose delta is n rows: of the first variable alone (where it keeps more), and of the first two."""
    out = []
    for a in {n, n // 2}:
        b = n - a
        if 2 * a < sizes[0] and 2 * b < sizes[1]:
            m = [np.ones(d, bool) for d in sizes]
            m[0][:a] = False
            m[1][sizes[1] - b:] = False
            out.append(m)
    return out


@pytest.mark.parametrize("t,opt", [(9_000, {}), (60_000, {}), (60_000, {"no_split": 1}), (700_000, {})])
def test_calls_of_n_rows_match_the_oracle(t, opt):
    torch_cuda()
    sizes = [40, 37, 64]
    g = np.random.default_rng(t)
    tup = np.stack([g.integers(0, d, t) for d in sizes], axis=1).astype(np.int32)
    tup[: 40 * 37] = np.array([(i, j, (i * 7 + j) % 64) for i in range(40) for j in range(37)])  # every value supported
    gt = GpuTable([0] * 3, sizes, tup, opt=C.make_options(**opt))
    assert compare_call(gt, tup, [np.ones(d, bool) for d in sizes])[0] == O.OK
    level, seen = gt.save(), 0
    for n in ROWS:
        for m in _cuts(sizes, n):
            assert compare_call(gt, tup, m)[0] == O.OK
            assert gt.stats()["rows_ored"] == n
            seen += 1
            gt.restore(level)
            level = gt.save()
    assert seen >= len(ROWS)
    gt.close()


@pytest.mark.parametrize("t", [900, 9_000])
def test_network_updates_of_n_rows_match_the_oracle(t):
    torch = torch_cuda()
    sizes = [40, 37, 64]
    g = np.random.default_rng(t)
    tup = np.stack([g.integers(0, d, t) for d in sizes], axis=1).astype(np.int32)
    st, m = C.ct_model_create([0] * 3, sizes, stream=torch.cuda.current_stream())
    assert st == C.CT_OK and C.ct_model_add_table(m, [0, 1, 2], tup) >= 0
    words = int(C.dom_layout(sizes)[0][-1])
    assert C.ct_model_propagate(m) == C.CT_OK
    root = C.words_to_masks(C.ct_model_get_domains(m, words)[1], sizes)
    for n in ROWS:
        for cut in _cuts(sizes, n):
            new = [a & b for a, b in zip(root, cut)]
            st, out, _ = O.gac_table(tup, [0] * 3, new)
            st2, level = C.ct_model_save(m)
            assert st2 == C.CT_OK and C.ct_model_set_domains(m, C.masks_to_words(new)) == C.CT_OK
            assert C.ct_model_propagate(m) == st
            if st == O.OK:
                assert np.array_equal(C.ct_model_get_domains(m, words)[1], C.masks_to_words(out))
            assert C.ct_model_restore(m, level) == C.CT_OK
    C.ct_model_destroy(m)
