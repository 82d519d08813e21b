"""GPU parity of a table's construction: the supports rows and currTable built
from the tuple list equal their definition (row (i, v) holds tuple j iff its
i-th component is v or a wildcard, Sec. 2; tuples outside the domains dropped,
input order kept) at the edges of words, chunks, tiles of 1,024 tuples, and of
the 360 rows a block holds at once.
"""
import numpy as np
import pytest

from oracle import ct_oracle as O
from paper_2507_18413_gb300 import ct as C
from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


def _pack(bits):
    words = np.zeros((len(bits) + 31) // 32 * 4, np.uint8)
    packed = np.packbits(bits, bitorder="little")
    words[: len(packed)] = packed
    return words.view("<u4")


@pytest.mark.parametrize("sizes,t,stars,outside", [
    ([3, 1, 5], 1, 0.0, 0.0),
    ([7, 9], 31, 0.0, 0.0),
    ([7, 9], 33, 0.3, 0.0),
    ([32, 33, 2], 1_023, 0.0, 0.0),
    ([32, 33, 2], 1_024, 0.0, 0.2),
    ([32, 33, 2], 1_025, 0.1, 0.2),
    ([359, 360, 361], 4_099, 0.05, 0.0),
    ([65_536, 2], 3_000, 0.0, 0.01),
    ([5] * 70, 2_049, 0.02, 0.0),
    ([40, 24], 200_003, 0.0, 0.0),
])
def test_rows_and_currtable_match_their_definition(sizes, t, stars, outside):
    torch_cuda()
    g = np.random.default_rng(t + len(sizes))
    lo = [int(v) for v in g.integers(-50, 50, len(sizes))]
    tup = np.stack([g.integers(0, d, t) + l for d, l in zip(sizes, lo)], axis=1).astype(np.int32)
    tup[g.random(tup.shape) < stars] = C.CT_STAR
    bad = g.random(t) < outside
    tup[bad, 0] = lo[0] + sizes[0]
    kept = tup[~bad]
    st, h = C.ct_create(len(sizes), lo, sizes, tup)
    assert st == C.CT_OK, C.last_error()
    info = C.ct_get_info(h)[1]
    nw = (len(kept) + 31) // 32
    assert info["tuples"] == len(kept) and info["words"] == nw
    assert info["short_tuples"] == int((kept == C.CT_STAR).any(axis=1).sum())
    st, table, nz = C.ct_get_currtable(h, nw)
    assert np.array_equal(table, O.currtable_words(np.ones(len(kept), bool))) and nz == nw
    assert C.ct_get_index(h)[1].tolist() == list(range((nw + 3) // 4))
    row = 0
    for i, d in enumerate(sizes):
        picks = range(d) if d <= 64 else sorted({0, 1, d // 2, 358, 359, 360, d - 2, d - 1} & set(range(d)))
        for v in picks:
            st, got = C.ct_get_support_row(h, row + v, nw)
            assert st == C.CT_OK
            want = _pack((kept[:, i] == lo[i] + v) | (kept[:, i] == C.CT_STAR))
            assert np.array_equal(got, want[:nw]), (i, v)
        row += d
    C.ct_destroy(h)


def test_a_list_outside_the_domains_is_infeasible():
    torch_cuda()
    st, h = C.ct_create(2, [0, 0], [4, 4], np.array([[4, 0], [-1, 2], [2**31 - 1, 0], [-2**31 + 1, 1]], np.int32))
    assert st == C.CT_INFEASIBLE and h
    C.ct_destroy(h)
