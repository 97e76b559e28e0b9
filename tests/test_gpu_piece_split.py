"""Table pieces of a cloud large enough for one warp per small piece: cells of 1 to
1100 points, so that pieces lie on both sides of the sizes where a warp, a block
and the split tree hand over, under leaves two or three levels above the cells
(tables of three and of four levels), against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import assert_build_matches_oracle, dev_points

pytestmark = pytest.mark.gpu

N = (1 << 25) + 4099


# a level-4 node holds 142,800 points on average: some are leaves, some are not
@pytest.mark.parametrize("s,lmax,C", [(7, 15, 142_800)])
def test_split_pieces(gpu_lib, s, lmax, C):
    fp = gpu_lib
    rng = np.random.default_rng(s + lmax)
    # 128 x 128 x 8 cells of the level-7 grid, of sizes that climb from 1 to 1100 and some empty
    sizes = np.tile([1, 31, 32, 33, 64, 96, 127, 128, 129, 200, 256, 257, 512, 1024, 1025, 1100, 0, 5], 8000)
    sizes = sizes[: int(np.searchsorted(np.cumsum(sizes), N))]
    sizes[-1] += N - int(sizes.sum())
    cell = np.repeat(np.arange(len(sizes)), sizes)
    w = 1 << 14   # the side of a cell of 2^21
    pts = np.zeros(N, synth.POINT_DTYPE)
    for a, c in (("x", cell % 128), ("y", (cell // 128) % 128), ("z", cell // 16384)):
        pts[a] = c * w + rng.integers(0, w, N)
    for a in "xyz":
        pts[a][0], pts[a][1] = 0, (1 << 21) - 1
    pts = pts[rng.permutation(N)]
    r = fp.build_octree(dev_points(pts), fp.params(7, s, lmax, 16, 1 << 20, C))
    torch.cuda.synchronize()
    assert fp.get_device_error() == 0
    want = oracle.build_all(pts, oracle.params(7, s, lmax, 16, 1 << 20, C))
    M = int(r["num_nodes"].item())
    assert_build_matches_oracle(want, cube=r["cube"], nodes=r["nodes"][:M], final=r["final"],
                                final_perm=r["final_perm"])
