"""The kernels that find every point's level-of-detail owner, at the sizes where
one hands over to the next: cells of 1 .. 32 points (pairs), 33 .. 1024 (tables,
with 256 and 512 as the edges of their variants), more (split first), at every
depth below the cell from none to beyond the tables (4 levels direct, 10 levels
hashed), with points spread through the cell, on a plane, on a line and on one
spot; and the count grid's two passes at every grid level, with empty octants and
thresholds from one point to the whole cloud.  Everything against the oracle,
element by element (integer work: no tolerance)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import assert_build_matches_oracle, dev_points

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 32, 33, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2500]
SIDE = 1 << 21


def cells_cloud(spread, seed, sizes=SIZES):
    """One level-3 cell of every size, points in random order; two far corners fix the cube."""
    rng = np.random.default_rng(seed)
    w = SIDE >> 3
    rows = [np.array([[0, 0, 0], [SIDE - 1] * 3])]
    for k, n in enumerate(sizes):
        m = 9 + 17 * k   # cells apart from each other and from the corners'
        base = np.array([(m >> 6) & 7, (m >> 3) & 7, m & 7]) * w
        p = rng.integers(0, w, (n, 3))
        if spread == "plane":
            p[:, 2] = p[:, 0] // 2
        elif spread == "line":
            p[:, 1:] = p[:, :1]
        elif spread == "spot":
            p = p[:1] + rng.integers(0, 3, (n, 3))
            p = np.minimum(p, w - 1)
        rows.append(base + p)
    xyz = np.concatenate(rows)
    xyz = xyz[rng.permutation(len(xyz))]
    pts = np.zeros(len(xyz), synth.POINT_DTYPE)
    pts["x"], pts["y"], pts["z"] = xyz.T
    pts["r"] = np.arange(len(xyz)) & 255
    return pts


def check(fp, pts_np, g, s, lmax, T, C):
    r = fp.build_octree(dev_points(pts_np), fp.params(g, s, lmax, 16, T, C))
    torch.cuda.synchronize()
    assert fp.get_device_error() == 0
    want = oracle.build_all(pts_np, oracle.params(g, s, lmax, 16, T, C))
    K = len(want["offsets"]) - 1
    assert int(r["num_chunks"].item()) == K
    assert np.array_equal(r["offsets"].cpu().numpy().view(np.uint64)[:K + 1], want["offsets"])
    assert np.array_equal(r["lut"].cpu().numpy().view(np.uint32), want["lut"])
    M = int(r["num_nodes"].item())
    assert_build_matches_oracle(want, cube=r["cube"], nodes=r["nodes"][:M], final=r["final"],
                                final_perm=r["final_perm"])


# depth of the decision below a level-3 cell whose leaf is the root: s - 4 levels
@pytest.mark.parametrize("spread", ["volume", "plane", "line", "spot"])
@pytest.mark.parametrize("s", [3, 4, 5, 7, 8, 9, 13, 14, 15, 18])
def test_piece_sizes_and_depths(gpu_lib, spread, s):
    check(gpu_lib, cells_cloud(spread, s), 3, s, 4, 1 << 20, 1 << 20)


# leaves below the cells: inner pieces, split nodes, owners at several levels
@pytest.mark.parametrize("spread", ["volume", "plane", "line", "spot"])
@pytest.mark.parametrize("s,lmax,C", [(3, 12, 20), (7, 15, 300), (5, 9, 1000), (11, 11, 40)])
def test_pieces_below_leaves(gpu_lib, spread, s, lmax, C):
    check(gpu_lib, cells_cloud(spread, 7 * s + C), 3, s, lmax, 2000, C)


# split rounds: nodes of one tile (4096 records) and of several, split again and again where
# the points lie close together, down to runs of equal keys; leaves above and below the cells
@pytest.mark.parametrize("spread", ["volume", "plane", "line", "spot"])
@pytest.mark.parametrize("s,lmax,C", [(7, 15, 1 << 20), (7, 15, 3000), (10, 12, 700), (3, 18, 50), (5, 8, 5000)])
def test_split_rounds(gpu_lib, spread, s, lmax, C):
    sizes = [1025, 4095, 4096, 4097, 8193, 30_000, 70_000]
    check(gpu_lib, cells_cloud(spread, 3 * s + lmax, sizes), 3, s, lmax, max(C, 20_000), C)


# more nodes than the one-launch node table takes, and as few as one
@pytest.mark.parametrize("n,g,s,lmax,C", [(60_000, 4, 5, 15, 1), (1, 4, 5, 15, 1), (60_000, 7, 7, 15, 1 << 20)])
def test_node_counts(gpu_lib, n, g, s, lmax, C):
    check(gpu_lib, synth.lidar(n, 77), g, s, lmax, max(C, 2000), C)


@pytest.mark.parametrize("g", [1, 2, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("T,C", [(1, 1), (40, 7), (3000, 500), (1 << 20, 1 << 20)])
def test_grid_passes(gpu_lib, g, T, C):
    pts = synth.uniform(6_000, 60 + g, bits=18)
    pts["x"][:3_000] //= 4      # a dense slab and an empty one
    pts["y"][3_000:] |= 1 << 17
    check(gpu_lib, pts, g, 7, 8, T, C)
