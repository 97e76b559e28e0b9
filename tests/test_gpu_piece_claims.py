"""Table pieces taken by the blocks one at a time (fewer than 32 pieces a block:
the first claim is followed at once by the next), at the numbers of pieces where a
block goes from none to one to two pieces and where the claims get longer, on 1520
resident blocks.  Every output against the oracle (whole numbers: no tolerance)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import assert_build_matches_oracle, dev_points

pytestmark = pytest.mark.gpu

BLOCKS = 152 * 10
G = 6


def pieces_cloud(pieces, seed):
    """A level-6 cell of 33 to 36 points for every piece, two far corners, random order."""
    rng = np.random.default_rng(seed)
    w = 1 << 14   # the side of a cell of 2^20
    cell = rng.choice((1 << (3 * G)) - 2, pieces, replace=False) + 1
    at = np.repeat(cell, 33 + np.arange(pieces) % 4)
    pts = np.zeros(len(at) + 2, synth.POINT_DTYPE)
    for k, a in enumerate("xyz"):
        pts[a][:-2] = ((at >> (G * k)) & ((1 << G) - 1)) * w + rng.integers(0, w, len(at))
        pts[a][-1] = (1 << 20) - 1
    return pts[rng.permutation(len(pts))]


@pytest.mark.parametrize("pieces", [1, BLOCKS - 1, BLOCKS, BLOCKS + 1, 2 * BLOCKS + 1, 32 * BLOCKS - 1, 32 * BLOCKS])
def test_single_claims(gpu_lib, pieces):
    fp = gpu_lib
    pts = pieces_cloud(pieces, pieces)
    prm = (G, 9, 12, 16, 1 << 21, 1 << 21)
    want = oracle.build_all(pts, oracle.params(*prm))
    dev = dev_points(pts)
    for _ in range(3):
        r = fp.build_octree(dev, fp.params(*prm))
        torch.cuda.synchronize()
        assert fp.get_device_error() == 0
        M = int(r["num_nodes"].item())
        assert_build_matches_oracle(want, cube=r["cube"], nodes=r["nodes"][:M], final=r["final"],
                                    final_perm=r["final_perm"])
