"""Scratch of weighted builds: their border lists hold at most one entry a
point, beside staging that holds one record a point twice."""
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


def test_border_lists_one_entry_a_point(lod):
    # Eight leaves of the root with all points in the cells beside the middle
    # planes, so that all of them are border entries.  A filtered build of the
    # same cloud differs in its scratch by two levels of 16-byte sums (32 bytes a
    # point) where the weighted one has the lists (16 bytes a point) and 16 bytes
    # a node; every block is rounded to 2 MB.
    import torch
    n = 1_000_000
    rng = np.random.default_rng(5)
    pts = np.empty((n, 4), np.int32)
    pts[:, :3] = rng.integers(0, 1 << 14, (n, 3))
    pts[:, 0] = (1 << 13) + rng.integers(-64, 64, n)
    pts[:2, :3] = [[0, 0, 0], [(1 << 14) - 1] * 3]
    pts[:, 3] = rng.integers(-(2**31), 2**31, n)
    d = torch.from_numpy(pts).cuda()
    held = {}
    for mode in (0, 2):
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        r = lod.build(d, 200_000, mode, 1, stream=st)
        held[mode] = lod.scratch_bytes(st)
        compare(r.to_host(stream=st), oracle.build(pts, 200_000, mode, 1), inp=pts)
        r.free()
        lod.trim(st)
    assert held[2] <= held[0] - 32 * n + 16 * n + 2 * (2 << 20)
