"""Size of the voxel array: its first size is held to a few records a point on
clouds whose nodes stand above one another, where the number of voxels cannot
be told from the node counts; a build that has no memory for it makes do with
less."""
import ctypes

import numpy as np
import pytest

import oracle
from compare import compare
from paper_2302_14801_gb300 import synth

pytestmark = pytest.mark.gpu

NODE, POINT, VOXEL = 56, 16, 16


@pytest.fixture(scope="module")
def lod():
    import torch
    from paper_2302_14801_gb300 import _build_ext
    _build_ext.build()
    from paper_2302_14801_gb300 import lod as m
    torch.cuda.set_device(0)
    return m


class Pool:
    """The device's default stream-ordered pool, which holds the results."""
    USED, USED_HIGH = 7, 8  # cudaMemPoolAttrUsedMemCurrent, cudaMemPoolAttrUsedMemHigh

    def __init__(self):
        import torch
        try:
            self.rt = ctypes.CDLL("libcudart.so.13")
        except OSError:
            pytest.skip("CUDA runtime library not found by name")
        self.pool = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.pool), torch.cuda.current_device()) == 0

    def read(self, attr):
        val = ctypes.c_uint64()
        assert self.rt.cudaMemPoolGetAttribute(self.pool, attr, ctypes.byref(val)) == 0
        return val.value

    def peak_of(self, call):
        """What call() returns, and the most bytes in use meanwhile beyond those before."""
        import torch
        torch.cuda.synchronize()
        zero = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolSetAttribute(self.pool, self.USED_HIGH, ctypes.byref(zero)) == 0
        base = self.read(self.USED)
        out = call()
        torch.cuda.synchronize()
        return out, self.read(self.USED_HIGH) - base


def clusters(n, each, chain):
    """Clusters of `each` points, identical ones, or (chain) identical but for a
    point at 1, 2, 4 ... from them, so that every node above has two children."""
    rng = np.random.default_rng(n + each)
    k = n // each
    at = rng.choice(1 << 18, k, replace=False)
    base = np.stack([at & 63, (at >> 6) & 63, at >> 12], 1) << 16
    xyz = np.repeat(base[:, None], each, axis=1)
    if chain:
        xyz[:, :16, 0] += 1 << np.arange(16)
    pts = np.empty((n, 4), np.int32)
    pts[:, :3] = xyz.reshape(-1, 3)
    pts[:, 3] = rng.integers(-(2**31), 2**31, n)
    return pts


def first_voxels(n, T):
    return max(n // 2, 4096, int(n * min(4.0, 20480 / T)))


@pytest.mark.parametrize("chain", [False, True])
@pytest.mark.parametrize("T,each", [(1000, 5000), (20_000, 50_000)])
def test_first_size_is_a_few_records_a_point(lod, T, each, chain):
    import torch
    n = 1_000_000
    pts = clusters(n, each, chain)
    d = torch.from_numpy(pts).cuda()
    want = oracle.build(pts, T, 0)
    r, peak = Pool().peak_of(lambda: lod.build(d, T, 0))
    got = r.to_host()
    r.free()
    compare(got, want, inp=pts)
    nodes = 64 + 16 * -(-n // T)
    while nodes < len(want["level"]):
        nodes *= 4
    # the result at the array's first size, its trimmed copy, and 1 MB for rounding
    assert peak <= n * POINT + nodes * NODE + (first_voxels(n, T) + len(want["voxels"])) * VOXEL + (1 << 20)


@pytest.mark.parametrize("mode", [0, 1])
def test_no_memory_for_the_first_size(lod, mode, monkeypatch):
    # the k-th device allocation of the build fails (on the host, never asked of
    # CUDA).  The voxel array's first one, here more than half a record a point,
    # is asked for again with less, and its trimmed copy done without; the ones
    # before them are not, nor are the picked points after them
    import torch
    pts = synth.indoor(400_000, seed=41, n_prims=64)
    want = oracle.build(pts, 3000, mode, 21)
    assert len(want["voxels"]) > len(pts) // 2  # the levels run twice with less
    d = torch.from_numpy(pts).cuda()
    pool, built = Pool(), []
    lod.build(d, 3000, mode).free()
    torch.cuda.synchronize()
    base = pool.read(Pool.USED)
    for k in range(1, 64):
        monkeypatch.setenv("LOD_INJECT_OOM_AT", str(k))
        try:
            r = lod.build(d, 3000, mode, full_precision=mode == 1)
        except lod.LodError as e:
            assert e.status == lod.LOD_ERR_OOM
            torch.cuda.synchronize()
            assert pool.read(Pool.USED) == base
            continue
        monkeypatch.delenv("LOD_INJECT_OOM_AT")
        built.append(k)
        compare(r.to_host(), want, inp=pts)
        r.free()
    first = built[0]
    if mode == 1:
        assert built != list(range(first, 64))  # a later failure is a failure
    monkeypatch.setenv("LOD_INJECT_OOM_AT", str(first))
    r = lod.build(d, 3000, mode)
    monkeypatch.delenv("LOD_INJECT_OOM_AT")
    nodes = r.device_bytes() - len(pts) * (POINT + 4 * mode) - len(want["voxels"]) * VOXEL
    r.free()
    assert nodes in [(64 + 16 * 134) * NODE * 4**j for j in range(3)]  # the second run left the exact size


@pytest.mark.parametrize("cloud,T", [("indoor", 3000), ("indoor", 1000), ("aerial", 3000), ("sphere", 1000)])
@pytest.mark.parametrize("full", [False, True])
def test_results_keep_little_slack(lod, cloud, T, full):
    # a result holds at most half a record a point, or half as many more records
    # than voxels (and 65536, below which nothing is copied); its picked points
    # at full precision are as many as its voxels
    import torch
    n = 3_000_000
    pts = getattr(synth, cloud)(n, seed=1)
    r = lod.build(torch.from_numpy(pts).cuda(), T, 1 if full else 0, full_precision=full)
    v = r.view().n_voxels
    extra = r.device_bytes() - n * (POINT + 4 * full) - v * VOXEL * full
    r.free()
    nodes = 64 + 16 * -(-n // T)
    assert extra <= nodes * NODE + max(n // 2, v + v // 2 + 65536) * VOXEL


def test_out_of_core_batches_keep_little(lod):
    # eight chunks in several batches, whose arrays all stay until the merge of
    # the root: a first size of four records a point must not stay with them,
    # nor sums beside it
    n, T, batch = 1_000_000, 1000, 250_000
    pts = clusters(n, 5000, True)
    want = oracle.build(pts, T, 0)
    r, peak = Pool().peak_of(lambda: lod.build_out_of_core(pts, T, 0, 21, chunk_points=n // 2, stream_points=batch, batch_points=batch))
    compare(r.to_host(), want, inp=pts)
    r.free()
    nodes = 8 * 64 + 16 * (n // T + 8)
    # every chunk's points, nodes and voxels with their sums, one batch's input
    # (points and indices) and first size, the counts of the top grid's 256^3
    # cells, the merge's grid (40 bytes for each of 128^3 cells), the assembled result
    most = (2 * (n * POINT + nodes * NODE + len(want["voxels"]) * 2 * VOXEL)
            + batch * (POINT + 4) + first_voxels(batch, T) * VOXEL + 4 * 256**3 + 40 * 128**3)
    assert peak <= most + (4 << 20)


def test_server_keeps_to_its_budget(lod):
    # the smallest budget that takes the request leaves half a record a point for
    # the voxel array; a large one lets it start at four, and the result keeps
    # no slack either way
    import torch
    n, T = 1_000_000, 1000
    pts = clusters(n, 5000, True)
    d = torch.from_numpy(pts).cuda()
    want = oracle.build(pts, T, 0)
    nodes = 64 + 16 * (n // T)

    def serve(budget):
        srv = lod.Server(hbm_budget_bytes=budget, max_inflight=1)
        try:
            try:
                ticket = srv.submit(d, T, 0)
            except lod.LodError as e:
                assert e.status == lod.LOD_ERR_BUDGET
                return None
            return srv.wait(ticket)
        finally:
            srv.close()

    refused, taken = 1 << 20, 1 << 30
    assert serve(refused) is None
    while taken - refused > 1:
        mid = (refused + taken) // 2
        r = serve(mid)
        if r is None:
            refused = mid
        else:
            taken = mid
            r.free()
    for budget, records in ((taken, n // 2), (8 << 30, first_voxels(n, T))):
        r, peak = Pool().peak_of(lambda: serve(budget))
        compare(r.to_host(), want, inp=pts)
        size = r.device_bytes()
        r.free()
        assert size == n * POINT + nodes * NODE + len(want["voxels"]) * VOXEL
        assert peak <= n * POINT + nodes * NODE + (records + len(want["voxels"])) * VOXEL + (1 << 20)


@pytest.mark.parametrize("cloud", ["indoor", "sphere"])
def test_server_results_keep_no_slack(lod, cloud):
    import torch
    n, T = 1_000_000, 1000
    d = torch.from_numpy(getattr(synth, cloud)(n, seed=1)).cuda()
    srv = lod.Server(hbm_budget_bytes=8 << 30, max_inflight=1)
    try:
        r = srv.wait(srv.submit(d, T, 0))
        v = r.view().n_voxels
        assert v > n // 2
        assert r.device_bytes() == n * POINT + (64 + 16 * (n // T)) * NODE + v * VOXEL
        r.free()
    finally:
        srv.close()
