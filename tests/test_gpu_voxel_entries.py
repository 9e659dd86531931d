"""Edges of the voxel pass's shared-memory entries, against the CPU oracle
(integer results, so the tolerance is equality): 16-bit colour fields that
wrap, keys that share their high word, ranks beyond 16 bits."""
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


def check(lod, pts, T, mode, max_depth=21):
    import torch
    r = lod.build(torch.from_numpy(pts).cuda(), T, mode, max_depth)
    got = r.to_host()
    r.free()
    compare(got, oracle.build(pts, T, mode, max_depth), inp=pts)


def in_octants(cells, rgba, octant, other=1):
    """Points at the given cells (x, y, z in 0..63) of one octant of a root
    cube of edge 128 (so a point is a cell), and `other` points far away."""
    k = np.array([(octant >> 2) & 1, (octant >> 1) & 1, octant & 1])
    pts = np.empty((len(cells) + other + 2, 4), np.int32)
    pts[:len(cells), :3] = np.asarray(cells) + 64 * k
    pts[:len(cells), 3] = rgba
    pts[len(cells):, :3] = 64 * (1 - k) + 5
    pts[len(cells):, 3] = 0x01020304
    pts[-2:, :3] = [[0, 0, 0], [127, 127, 127]]
    return pts


@pytest.mark.parametrize("n", [256, 257, 258, 514, 30_000, 65_535, 65_536, 70_000])
@pytest.mark.parametrize("rgba", [-1, 0x0000FF00, 0x00FF01FF])
def test_colour_fields_that_wrap(lod, n, rgba):
    # one cell of n points of one colour (255 * 257 = 65,535 is the largest
    # 16-bit sum), two smaller ones beside it, in one leaf of the root;
    # 65,535 points is the largest leaf the 16-bit layout takes
    cells = np.repeat([[3, 4, 5], [4, 4, 5], [63, 63, 63]], [n - n // 3 - 1, n // 3, 1], axis=0)
    check(lod, in_octants(cells, rgba, 5, other=2), n + 1, 0, max_depth=1)


def splitmix64(x):
    with np.errstate(over="ignore"):
        z = x.astype(np.uint64) + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


@pytest.mark.parametrize("mode", [1, 4])
def test_keys_that_share_their_high_word(lod, mode):
    # pairs of input indices whose keys agree in the upper 32 bits, each pair
    # alone in a cell: pick keys by collision, random keys (12 bits above the
    # low 20 bits of the index) from indices 2^20 apart
    n = 400_000 if mode == 1 else (1 << 20) + 300_000
    ix = np.arange(n)
    if mode == 1:
        hi = (splitmix64(ix) >> np.uint64(32)).astype(np.int64)
        order = np.argsort(hi, kind="stable")
        same = np.nonzero(hi[order][1:] == hi[order][:-1])[0]
        pairs = np.stack([order[same], order[same + 1]], 1)
    else:
        r = (splitmix64(ix) >> np.uint64(52)).astype(np.int64)  # level 0: the root's grid
        a = ix[:300_000]
        a = a[r[a] == r[a + (1 << 20)]]
        pairs = np.stack([a, a + (1 << 20)], 1)
    assert len(pairs) >= 5
    rng = np.random.default_rng(7)
    cells = rng.integers(0, 32, (n, 3))
    cells[:, 2] += 32  # everything else in the octant's upper half
    for j, (a, b) in enumerate(pairs[:1000]):
        cells[a] = cells[b] = [j % 32, j // 32, 1]
    rgba = rng.integers(-(2**31), 2**31, n)
    pts = np.empty((n + 2, 4), np.int32)
    pts[:n, :3], pts[:n, 3] = cells, rgba
    pts[n:] = [[0, 0, 0, 5], [127, 127, 127, 6]]
    check(lod, pts, n // 2, mode, max_depth=1)


@pytest.mark.parametrize("mode", [0, 1, 3, 4])
def test_ranks_beyond_16_bits(lod, mode):
    # leaves of 200,000 points with about 140,000 occupied cells each: more
    # than the 16-bit word ranks count from the octant's first cell
    rng = np.random.default_rng(11)
    pts = np.empty((1_600_000, 4), np.int32)
    pts[:, :3] = rng.integers(0, 1 << 14, (1_600_000, 3))
    pts[:, 3] = rng.integers(-(2**31), 2**31, 1_600_000)
    check(lod, pts, 300_000, mode, max_depth=1)


@pytest.mark.parametrize("depth", [1, 2, 3])
@pytest.mark.parametrize("L", [2, 6, 7, 8, 9, 15, 31, 32])
def test_weighted_samples_across_octants(lod, L, depth):
    # points within two cells of the middle planes of a cube of edge 2^L, on
    # one, two or all three axes: their weights reach one to seven siblings;
    # deeper trees hand voxels across the planes as well
    rng = np.random.default_rng(100 * L + depth)
    n, mid, cell = 3000, 1 << (L - 1), max(1, (1 << L) >> 7)
    p = rng.integers(0, 1 << L, (n, 3))
    near = rng.random((n, 3)) < 0.6
    p = np.where(near, mid + rng.integers(-2 * cell, 2 * cell + 1, (n, 3)), p)
    p[:3] = mid
    p[3:6] = mid - 1
    p[6:8] = [[0, 0, 0], [(1 << L) - 1] * 3]
    p = np.clip(p, 0, (1 << L) - 1) - (1 << 31 if L == 32 else 0)
    pts = np.empty((n, 4), np.int32)
    pts[:, :3] = p
    pts[:, 3] = rng.integers(-(2**31), 2**31, n)
    check(lod, pts, 20, 2, max_depth=depth)


@pytest.mark.parametrize("mode", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("tiles", [1, 2, 3, 4, 5, 9, 10])
def test_levels_of_few_items(lod, mode, tiles):
    # 8 to 80 items at the top level: clusters of 8, 4 and 2 CTAs, and none;
    # leaves (with kept indices) and inner children beside each other
    import torch
    rng = np.random.default_rng(17 * tiles + mode)
    clouds = []
    for t in range(tiles):
        n = 9001 + 700 * t
        pts = np.empty((n, 4), np.int32)
        pts[:, :3] = rng.integers(0, 1 << 12, (n, 3))
        pts[: n // 3, :3] >>= 2
        pts[:2, :3] = [[0, 0, 0], [(1 << 12) - 1] * 3]
        pts[:, 3] = rng.integers(-(2**31), 2**31, n)
        clouds.append(pts)
    rs = lod.build_batched([torch.from_numpy(c).cuda() for c in clouds], 1500, mode, keep_index=True)
    for c, r in zip(clouds, rs):
        compare(r.to_host(), oracle.build(c, 1500, mode, 21), inp=c)
        r.free()
