"""The node table by a cluster of CTAs (room for 32768 nodes a tile or more)
and by one CTA, against the oracle."""
import numpy as np
import pytest

import oracle
from compare import compare
from test_gpu_parity import gpu_build, lod  # noqa: F401

pytestmark = pytest.mark.gpu


def _cube(n, bits, seed):
    rng = np.random.default_rng(seed)
    pts = np.empty((n, 4), np.int32)
    pts[:, :3] = rng.integers(0, 1 << bits, size=(n, 3))
    pts[:, 3] = rng.integers(-(2**31), 2**31, size=n)
    return pts


# (points, T): one CTA; just over the line; levels of several steps of a cluster
@pytest.mark.parametrize("n,T", [(20_430, 10), (20_431, 10), (40_000, 7), (60_000, 2)])
def test_sizes(lod, n, T):  # noqa: F811
    pts = _cube(n, 18, n)
    compare(gpu_build(lod, pts, T, 0), oracle.build(pts, T, 0), inp=pts)


def test_capacity_overflow(lod):  # noqa: F811
    # chains of nodes with seven one-point leaves beside each: several times more
    # nodes than the table's first size has room for (16 per T points)
    T, bits = 100, 24
    off = [np.zeros((T + 1, 3), np.int64)]
    off += [np.array([[k >> 2, (k >> 1) & 1, k & 1] for k in range(1, 8)], np.int64) << lg for lg in range(3, bits - 4)]
    off = np.concatenate(off)
    g = np.arange(1000)
    base = np.stack([g & 15, (g >> 4) & 15, g >> 8], 1).astype(np.int64) << (bits - 4)
    xyz = np.concatenate([(base[:, None] + off[None]).reshape(-1, 3), np.full((1, 3), (1 << bits) - 1)])
    pts = np.empty((len(xyz), 4), np.int32)
    pts[:, :3] = xyz
    pts[:, 3] = np.arange(len(xyz))
    compare(gpu_build(lod, pts, T, 0), oracle.build(pts, T, 0), inp=pts)


def test_uneven_tiles(lod):  # noqa: F811
    import torch
    tiles = [_cube(n, 17, n) for n in (150_000, 1, 90_000)]  # a cluster each, the one-point tile's too
    rs = lod.build_batched([torch.from_numpy(t).cuda() for t in tiles], 2, 0)
    for t, r in zip(tiles, rs):
        compare(r.to_host(), oracle.build(t, 2, 0, 21), inp=t)
        r.free()
