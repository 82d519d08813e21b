"""GPU parity of the one-CTA kernel for small tables and of the general kernel at
the sizes where the choice between them lies (128 chunks, 512 values, 16
variables, 4 words per domain), positive, short and negative tables, through
both entry points, with backtracking; every call compared with the oracle.
"""
import numpy as np
import pytest

from oracle import ct_oracle as O
from oracle import negative as N
from oracle import short as S
from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G
from gpu_helpers import GpuTable, compare_call, torch_cuda

pytestmark = pytest.mark.gpu


def _edit(rng, masks, k):
    """Edits of one variable, or (every third) of all of them at once: row lists of several batches."""
    if k % 3 == 2:
        new = [m.copy() for m in masks]
        for m in new:
            v = np.flatnonzero(m)
            m[v[np.argsort(rng.u64(len(v)), kind="stable")[: len(v) // (2 + k % 2)]]] = False
        return new
    return (G.delta_step if rng.int(2) else G.reset_step)(rng, masks)[0]


@pytest.mark.parametrize("sizes,t,opt", [
    ([8, 8, 8], 200, {}),
    ([8, 8, 8], 1, {}),
    ([5, 6], 33, {}),
    ([128, 128, 128, 128], 16_384, {}),       # 128 chunks, 512 values, 4 words
    ([128, 128, 128, 127], 16_385, {}),       # 129 chunks
    ([128, 128, 128, 128, 1], 5_000, {}),     # 513 values
    ([129, 40], 3_000, {}),                   # 5 words
    ([6] * 16, 4_097, {}),
    ([6] * 17, 4_097, {}),
    ([40, 31, 20], 9_000, {"no_early_filter": 1}),
    ([40, 31, 20], 9_000, {"grid_blocks": 2}),
    ([40, 31, 20], 9_000, {"copy_state": 1}),
])
def test_positive_tables_match_the_oracle(sizes, t, opt):
    torch_cuda()
    g = np.random.default_rng(sum(sizes) + t)
    tup = np.stack([g.integers(0, d, t) for d in sizes], axis=1).astype(np.int32)
    lo = [0] * len(sizes)
    gt = GpuTable(lo, sizes, tup, opt=C.make_options(**opt) if opt else None)
    host = GpuTable(lo, sizes, tup, opt=C.make_options(**opt) if opt else None)
    full = [np.ones(d, bool) for d in sizes]
    st, root = compare_call(gt, tup, full)
    assert st == O.OK
    C.ct_propagate_host(host.h, C.masks_to_words(full))
    for x in (gt, host):
        x.save()
    rng, masks, fails = G.Rng(t), root, 0
    for k in range(30):
        for x in (gt, host):
            x.save()
        new = _edit(rng, masks, k)
        st, out = compare_call(gt, tup, new)
        w = C.masks_to_words(new)
        st_h, ch = C.ct_propagate_host(host.h, w, host.nch)
        assert st_h == st
        if st == O.OK:
            assert np.array_equal(w, C.masks_to_words(out))
            assert np.array_equal(host.currtable()[0], gt.currtable()[0])
        if st != O.OK or k % 7 == 6:
            fails += st != O.OK
            for x in (gt, host):
                x.restore(0)
                x.save()
            masks = root
        else:
            masks = out
    # domains that grew are refused, an empty one fails
    grown = [m.copy() for m in full]
    gt.restore(0)
    gt.save()
    if sizes[0] > 1:
        cut = [m.copy() for m in root]
        v = np.flatnonzero(cut[0])
        if len(v) > 1:
            cut[0][v[0]] = False
            st, out = compare_call(gt, tup, cut)
            if st == O.OK:
                back = [m.copy() for m in out]
                back[0][v[0]] = True
                assert gt.propagate(back)[0] == C.CT_ERR_STATE
    gt.restore(0)
    gt.save()
    grown[-1][:] = False
    assert gt.propagate(grown)[0] in (C.CT_INFEASIBLE, C.CT_ERR_STATE)
    gt.close()
    host.close()


@pytest.mark.parametrize("t,opt", [(700, {}), (16_400, {}), (700, {"grid_blocks": 3})])
def test_short_tables_match_the_oracle(t, opt):
    torch_cuda()
    sizes = [9, 30, 40, 17]
    tup = G.short_tuples(t, [0] * 4, sizes, t, 0.15)
    ret = S.retained_short(tup, [0] * 4, sizes)
    gt = GpuTable([0] * 4, sizes, tup, opt=C.make_options(**opt) if opt else None)
    masks = [np.ones(d, bool) for d in sizes]
    gt.save()
    rng = G.Rng(t)
    for k in range(16):
        gt.save()
        new = _edit(rng, masks, k)
        st_o, out, valid = S.gac_table_short(ret, [0] * 4, new)
        st, got, _ = gt.propagate(new)
        assert st == st_o
        if st == O.OK:
            assert all(np.array_equal(a, b) for a, b in zip(got, out))
            assert np.array_equal(gt.currtable()[0], O.currtable_words(valid))
            masks = out
        if st != O.OK or k % 5 == 4:
            gt.restore(0)
            gt.save()
            masks = [np.ones(d, bool) for d in sizes]
    gt.close()


@pytest.mark.parametrize("d,t,opt", [(7, 1_500, {}), (13, 20_011, {}), (7, 1_500, {"grid_blocks": 2})])
def test_negative_tables_match_the_oracle(d, t, opt):
    torch_cuda()
    sizes = [d, d, d, d + 1]
    tup = G.distinct_uniform_tuples(t, [0] * 4, sizes, t)
    st, h = C.ct_create(4, [0] * 4, sizes, tup, opt=C.make_options(**opt), negative=True)
    assert st == C.CT_OK, C.last_error()
    full = [np.ones(s, bool) for s in sizes]
    C.check(C.ct_save(h)[0])
    rng, masks, pruned = G.Rng(t), full, 0
    for k in range(30):
        C.check(C.ct_save(h)[0])
        new = _edit(rng, masks, k)
        st_o, out, valid = N.gac_table_negative(tup, [0] * 4, new)
        w = C.masks_to_words(new)
        st, _ = C.ct_propagate_host(h, w, 1)
        assert st == st_o or (st == C.CT_OK and any(not m.any() for m in out))  # (an emptied domain fails the next call)
        if st == C.CT_OK:
            assert np.array_equal(C.ct_get_currtable(h, (t + 31) // 32)[1], O.currtable_words(valid))
            assert np.array_equal(w, C.masks_to_words(out)), k
            pruned += any(not np.array_equal(a, b) for a, b in zip(out, new))
            masks = out
        if st != C.CT_OK or k % 6 == 5 or any(m.sum() < 2 for m in masks):
            C.check(C.ct_restore(h, 0))
            C.check(C.ct_save(h)[0])
            masks = full
    C.ct_destroy(h)
