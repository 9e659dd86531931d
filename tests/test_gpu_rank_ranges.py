"""Voxel items taken in several rank ranges on levels of too many items to be
shared by clusters, against the oracle: ranges that stay with the item's CTA,
and ranges handed to others (whether any were is read from the statistics of
LOD_DEBUG_STATS=1, so those builds run in a process of their own), with kept
indices and in every mode; octants of more than 65,535 occupied cells."""
import os
import re
import subprocess
import sys

import numpy as np
import pytest

import oracle
from compare import compare

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# (mode, kept indices) from the command line; marks each build in the statistics
SCRIPT = """
import sys
sys.path[:0] = ["tests"]
import torch
import oracle
from compare import compare
from paper_2302_14801_gb300 import lod, synth
mode, keep = int(sys.argv[1]), sys.argv[2] == "1"
pts = synth.indoor(300_000, seed=21, n_prims=64)
want = oracle.build(pts, 1000, mode, 21)
d = torch.from_numpy(pts).cuda()
for queue, cells in ((1, 97), (2, 97), (3, 97), (2, 500)):
    lod.set_tuning(vox_queue_ranges=queue, vox_range_cells=cells)
    print(f"[queue {queue}]", file=sys.stderr, flush=True)
    r = lod.build(d, 1000, mode, keep_index=keep)
    compare(r.to_host(), want, inp=pts)
    r.free()
"""


@pytest.mark.parametrize("mode,keep", [(0, 0), (0, 1), (1, 0), (2, 0), (2, 1), (3, 0), (4, 0)])
def test_ranges_handed_on(mode, keep):
    from paper_2302_14801_gb300 import _build_ext
    _build_ext.build()
    p = subprocess.run([sys.executable, "-c", SCRIPT, str(mode), str(keep)], cwd=ROOT,
                       env=dict(os.environ, LOD_DEBUG_STATS="1"), capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stderr[-2000:]
    builds = re.split(r"\[queue (\d)\]", p.stderr)[1:]
    assert builds[::2] == ["1", "2", "3", "2"]
    for queue, text in zip(builds[::2], builds[1::2]):
        levels = [(int(i), int(u)) for i, u in re.findall(r"items (\d+) .*queued ranges (\d+)", text)]
        # 152 SMs: levels of at most 76 items are shared by clusters, which queue nothing
        assert sum(i > 76 for i, _ in levels) >= 5
        assert all(u == 0 for i, u in levels if queue == "1" or i <= 76)
        assert queue == "1" or sum(u > 0 for _, u in levels) >= 3


@pytest.mark.parametrize("mode", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("tiles", [1, 10])
def test_octants_of_more_than_16_bits(mode, tiles):
    # one octant of 80,000 points in some 68,900 cells, a point or two in each of
    # the other seven: 8 items (a cluster each) or 80 (one CTA each, four ranges)
    import torch
    from paper_2302_14801_gb300 import _build_ext
    _build_ext.build()
    from paper_2302_14801_gb300 import lod
    clouds = []
    for t in range(tiles):
        rng = np.random.default_rng(10 * t + mode)
        pts = np.empty((80_009, 4), np.int32)
        pts[:80_000, :3] = rng.integers(0, 1 << 13, (80_000, 3)) + np.array([t & 1, (t >> 1) & 1, 1]) * (1 << 13)
        pts[80_000:, :3] = [[x, y, z] for x in (0, 16383) for y in (0, 16383) for z in (0, 16383)] + [[5, 5, 5]]
        pts[:, 3] = rng.integers(-(2**31), 2**31, 80_009)
        clouds.append(pts)
    rs = lod.build_batched([torch.from_numpy(c).cuda() for c in clouds], 80_005, mode, 1)
    for c, r in zip(clouds, rs):
        want = oracle.build(c, 80_005, mode, 1)
        assert len(want["voxels"]) > 65_535 + 8
        compare(r.to_host(), want, inp=c)
        r.free()
