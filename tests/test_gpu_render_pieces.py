"""The rasteriser's draw list at the edges of its pieces (2048 samples),
against the oracle rasteriser, bit for bit: leaves around whole pieces, inner
nodes of one to several pieces, many samples a pixel, points on the clip
volume's faces, with and without the counts."""
import numpy as np
import pytest

import oracle
from paper_2302_14801_gb300 import camera

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lod():
    import torch
    from paper_2302_14801_gb300 import _build_ext
    _build_ext.build()
    from paper_2302_14801_gb300 import lod as m
    torch.cuda.set_device(0)
    return m


@pytest.mark.parametrize("n", [1, 2047, 2048, 2049, 4096, 6145, 30_000])
@pytest.mark.parametrize("T", [2048, 100_000])
@pytest.mark.parametrize("pixels", [1e-3, 100.0, 1e6])
def test_pieces_equal_oracle(lod, n, T, pixels):
    import torch
    rng = np.random.default_rng(n)
    pts = np.empty((n, 4), np.int32)
    pts[:, :3] = rng.integers(0, 1 << 12, (n, 3))
    pts[:, 3] = rng.integers(-(2**31), 2**31, n)
    pts[: n // 4, :2] = pts[0, :2]  # a quarter of them behind one another
    lo, hi = pts[:, :3].min(0), pts[:, :3].max(0)
    want_res = oracle.build(pts, T, 0, 21)
    r = lod.build(torch.from_numpy(pts).cuda(), T, 0)
    # the box exactly (its corner points lie on the clip volume's faces), and
    # a box that cuts through the cloud
    for a, b in ((lo, np.maximum(hi, lo + 1)), (lo + (hi - lo) // 3, np.maximum(hi, lo + 1))):
        m, org = camera.orthographic(a, b)
        want, vis, drawn = oracle.render(want_res, m, org, 61, 37, pixels)
        fb, st = lod.render(r, m, org, 61, 37, pixels, stats=True)
        assert (st["visible_nodes"], st["samples_drawn"]) == (int(vis.sum()), drawn)
        assert np.array_equal(fb.cpu().numpy().view(np.uint64), want)
        assert torch.equal(lod.render(r, m, org, 61, 37, pixels), fb)
    r.free()
