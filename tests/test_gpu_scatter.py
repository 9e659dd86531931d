"""The scatter's leaf claims against the oracle where their tables run full or
stay nearly empty: more leaves in a CTA's share than its table holds, one leaf
for a whole share, leaves at every level of the first grid."""
import numpy as np
import pytest

import oracle
from compare import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lod():
    import torch
    from paper_2302_14801_gb300 import _build_ext
    _build_ext.build()
    from paper_2302_14801_gb300 import lod as m
    torch.cuda.set_device(0)
    return m


@pytest.mark.parametrize("n,T,cps,mode", [(1_500_000, 1, 1, 0), (400_000, 60, 1, 1), (700_000, 600_000, 2, 0), (700_001, 699_999, 0, 1)])
def test_leaf_claims(lod, n, T, cps, mode):
    import torch
    rng = np.random.default_rng(n + T)
    pts = np.empty((n, 4), np.int32)
    pts[:, :3] = rng.integers(0, 1 << 20, (n, 3))
    half = n // 2  # half of them thinned out towards a corner: leaves at many levels
    pts[:half, :3] = np.exp2(rng.uniform(0, 20, (half, 3))).astype(np.int64)
    pts[:, 3] = rng.integers(-(2**31), 2**31, n)
    want = oracle.build(pts, T, mode, 21)
    try:
        lod.set_tuning(stream_ctas_per_sm=cps)
        r = lod.build(torch.from_numpy(pts).cuda(), T, mode)
    finally:
        lod.set_tuning()
    got = r.to_host()
    r.free()
    compare(got, want, inp=pts)
