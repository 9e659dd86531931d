"""Page-locked host memory that a thread keeps between builds: bounded, and
given back by lod_trim.  The statistics line of LOD_DEBUG_STATS=1 reports it,
which the library reads once, so the builds run in a process of their own."""
import os
import re
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import torch
from paper_2302_14801_gb300 import lod
pts = torch.zeros((70_000, 4), dtype=torch.int32, device="cuda")
pts[:, 0] = torch.arange(70_000, device="cuda")
torch.cuda.synchronize()
for tiles in (1000, 70_000):  # 144 bytes a tile: 10 MB of tile tables in the second
    rs = lod.build_batched([pts[i:i + 1] for i in range(tiles)], 10, 0)
    assert all(r.view().n_points == 1 for r in rs)
    for r in rs:
        r.free()
lod.trim()
"""


def test_kept_bytes_are_bounded_and_trimmed():
    from paper_2302_14801_gb300 import _build_ext
    _build_ext.build()
    p = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, env=dict(os.environ, LOD_DEBUG_STATS="1"),
                       capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    kept = [int(x) for x in re.findall(r"host ms:.*page-locked bytes (\d+)", p.stderr)]
    # up to 8 MB each for uploads and read-backs; the second's read-backs are more
    assert len(kept) == 2 and 0 < kept[0] <= 16 << 20 and kept[1] <= 8 << 20
    assert re.findall(r"trim: page-locked bytes (\d+)", p.stderr) == ["0"]
