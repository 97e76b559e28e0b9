"""Trees split down to a few points: cells of 2 to 64 points whose node is inner, with
leaves one level below the cells and many, points spread, on a line and on one spot
(equal keys down to the last level), small inner pieces of the split rounds; every
node, owner and leaf against the oracle.  And a tree of a node a point does not take a
block per cell."""
import pytest
import torch

from tests.test_gpu_pieces import cells_cloud, check

pytestmark = pytest.mark.gpu

SMALL = [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 30, 31, 32, 33, 34, 63, 64]


@pytest.mark.parametrize("spread", ["volume", "plane", "line", "spot"])
@pytest.mark.parametrize("s,lmax,C", [(3, 4, 1), (3, 12, 1), (7, 15, 2), (3, 19, 7), (11, 11, 16), (4, 18, 31)])
def test_small_inner_cells(gpu_lib, spread, s, lmax, C):
    check(gpu_lib, cells_cloud(spread, 11 * s + C, SMALL), 3, s, lmax, max(C, 200), C)


# cells of more than 1024 points, split into inner pieces of any size
@pytest.mark.parametrize("spread", ["volume", "line", "spot"])
@pytest.mark.parametrize("s,lmax,C", [(3, 12, 1), (7, 15, 4), (5, 17, 20)])
def test_small_inner_pieces_of_splits(gpu_lib, spread, s, lmax, C):
    check(gpu_lib, cells_cloud(spread, 5 * s + C, [1025, 3000, 9000]), 3, s, lmax, max(C, 500), C)


LARGE = [33, 34, 100, 255, 256, 257, 512, 513, 1022, 1023, 1024]


# one block a piece: capacities at the ends of the sliding maximum's window (a power of two and beside it)
@pytest.mark.parametrize("spread", ["volume", "plane", "line", "spot"])
@pytest.mark.parametrize("s,lmax,C", [(3, 12, 1), (7, 15, 2), (5, 17, 31), (3, 19, 32), (9, 13, 255), (4, 4, 256), (6, 8, 1023)])
def test_large_inner_cells(gpu_lib, spread, s, lmax, C):
    check(gpu_lib, cells_cloud(spread, 13 * s + C, LARGE), 3, s, lmax, max(C, 1500), C)


def octree_ms(fp, pts, T, C):
    n = pts.shape[0]
    cube = fp.fp_bounds(pts)
    counts = fp.fp_count(pts, cube, 7)
    prm = fp.params(7, 7, 15, 16, T, C)
    chunks, num, lut, offsets = fp.fp_merge_chunks(counts, 7, T)
    dist, perm = fp.fp_distribute(pts, cube, 7, lut, offsets, num)
    ws = torch.empty(fp.workspace_size("octree", n, prm), dtype=torch.uint8, device="cuda")
    ms = []
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fp.fp_build_chunk_octree(dist, perm, cube, chunks, num, offsets, counts, prm, leaf=False, ws=ws)
        b.record()
        b.synchronize()
        ms.append(a.elapsed_time(b))
    assert fp.get_device_error() == 0
    return sorted(ms)[3]


def test_every_point_its_node(gpu_lib):
    """2 * 10^6 points at capacity 1 (2.9 * 10^6 nodes) take 7 times as long as at 20,000
    (73 times with a block for every cell of two points)."""
    pts = torch.randint(0, 1 << 20, (2_000_000, 4), dtype=torch.int32, device="cuda")
    assert octree_ms(gpu_lib, pts, 600, 1) < 15 * octree_ms(gpu_lib, pts, 20_000, 20_000)


def test_dense_cells_are_no_chain(gpu_lib):
    """Cells of up to 1024 points at capacity 2: 3.4 times as long as at 20,000 (11 times
    with their nodes found one after the other)."""
    pts = torch.randint(0, 1 << 20, (3_000_000, 4), dtype=torch.int32, device="cuda")
    for k in range(3):
        pts[:, k] = (torch.rand(3_000_000, device="cuda") ** 4 * (1 << 20)).to(torch.int32)
    a, b = octree_ms(gpu_lib, pts, 1000, 2), octree_ms(gpu_lib, pts, 20_000, 20_000)
    assert a < 6 * b, (a, b)
