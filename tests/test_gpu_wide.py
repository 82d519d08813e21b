"""GPU parity on wide tables: many values per table, domains of several words
(lanes sharing a variable in the plan and the publication), values probed one
per lane, tables whose windows cover every chunk (no full scan) and tables
whose undecided values are cut over the grid's warps. Every call is compared
bit-exactly with the oracle (status, domains, changed mask, currTable, index).
"""
import numpy as np
import pytest

from oracle import ct_oracle as O
from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G
from gpu_helpers import GpuTable, compare_call, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,t,opt", [
    ([150] * 40, 1_500, {}),               # global plan, 12 chunks: one window covers them
    ([150] * 40, 1_500, {"no_residues": 1}),  # ... every value by the full scan
    ([260] * 24, 16_500, {}),              # 129 chunks: one more than the windows cover
    ([97] * 7 + [600], 12_000, {}),        # local plan, one domain wider than the others
    ([70] * 12, 128 * 32 + 1, {"grid_blocks": 3}),  # few warps, several values each
    ([40_000, 30_000, 5], 5_000, {}),      # more domain words than a CTA stages
])
def test_wide_tables_match_the_oracle(sizes, t, opt):
    torch_cuda()
    g = np.random.default_rng(sum(sizes) + t)
    tup = np.stack([g.integers(0, d, t) for d in sizes], axis=1).astype(np.int32)
    lo = [0] * len(sizes)
    gt = GpuTable(lo, sizes, tup, opt=C.make_options(**opt) if opt else None)
    st, root = compare_call(gt, tup, [np.ones(d, bool) for d in sizes])
    assert st == O.OK
    gt.save()
    rng, masks, pruned = G.Rng(t), root, 0
    for k in range(14):
        gt.save()
        new, i = (G.delta_step if k % 3 == 1 else G.reset_step)(rng, masks)
        st, out = compare_call(gt, tup, new)
        pruned += gt.stats()["pruned"]
        if st != O.OK or k % 5 == 4:
            gt.restore(0)
            gt.save()
            masks = root
        else:
            masks = out
    assert pruned > 0
    gt.close()
