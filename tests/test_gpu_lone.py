"""The one-CTA-per-SM propagation against the general one on the same table, at
the size where the choice lies (a warp per segment and per value on one CTA per
SM) and just above the one-CTA kernel's range: domains, currTable and its index
after every call of a stream with backtracking.
"""
import numpy as np
import pytest

from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G
from gpu_helpers import GpuTable, torch_cuda

pytestmark = pytest.mark.gpu


def _edges(R):
    """Tuples of 128 chunks and one more, and of the segments that leave a warp per value and one more."""
    warps = 8 * torch_cuda().cuda.get_device_properties(0).multi_processor_count
    return [129 * 128, (warps - R) * 4096, (warps - R) * 4096 + 1]


@pytest.mark.parametrize("which", [0, 1, 2])
@pytest.mark.parametrize("sizes", [[32] * 6, [64, 33, 40, 128]])
def test_both_launch_shapes_agree(sizes, which):
    t = _edges(sum(sizes))[which]
    g = np.random.default_rng(t)
    tup = np.stack([g.integers(0, d, t, dtype=np.int32) for d in sizes], axis=1)
    lo = [0] * len(sizes)
    sms = torch_cuda().cuda.get_device_properties(0).multi_processor_count
    a, b = GpuTable(lo, sizes, tup), GpuTable(lo, sizes, tup, opt=C.make_options(grid_blocks=2 * sms))
    assert (a.info["grid_blocks"] <= sms) == (which < 2)
    root = [np.ones(d, bool) for d in sizes]
    rng, masks = G.Rng(t), root
    for k in range(14):
        for x in (a, b):
            x.save()
        new = (G.reset_step if k % 2 else G.delta_step)(rng, masks)[0]
        (sa, da, ca), (sb, db, cb) = a.propagate(new), b.propagate(new)
        assert sa == sb and np.array_equal(ca, cb)
        if sa != C.CT_OK or k % 6 == 5:
            for x in (a, b):
                x.restore(0)
            masks = root
            continue
        assert all(np.array_equal(x, y) for x, y in zip(da, db))
        (wa, na), (wb, nb) = a.currtable(), b.currtable()
        assert np.array_equal(wa, wb) and na == nb
        assert np.array_equal(np.sort(a.index()), np.sort(b.index()))
        masks = da
    a.close()
    b.close()
