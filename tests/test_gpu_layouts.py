"""The final layout and the leaf grouping at the sizes where one kernel hands over
to the next: one cluster (up to 2^15 points), one sort of the whole array (up to
2^21), the chunk-wise scatter above and, where a chunk holds more nodes than that
takes, the sort again; tiles of 1024 and 4096 records, one to four sort passes,
one chunk and thousands.  Everything against the oracle, element by element."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import assert_build_matches_oracle, assert_points_equal, dev_points

pytestmark = pytest.mark.gpu


def check(fp, pts_np, g, s, lmax, T, C):
    r = fp.build_octree(dev_points(pts_np), fp.params(g, s, lmax, 16, T, C))
    torch.cuda.synchronize()
    assert fp.get_device_error() == 0
    want = oracle.build_all(pts_np, oracle.params(g, s, lmax, 16, T, C))
    M = int(r["num_nodes"].item())
    assert_build_matches_oracle(want, cube=r["cube"], nodes=r["nodes"][:M], final=r["final"],
                                final_perm=r["final_perm"])
    assert np.array_equal(r["leaf_perm"].cpu().numpy().view(np.uint32), want["leaf_perm"])
    assert_points_equal(r["leaf_pts"], want["leaf_pts"])


@pytest.mark.parametrize("n", [1, 2, 1023, 1024, 1025, 8191, 8192, 8193, (1 << 15) - 1, 1 << 15, (1 << 15) + 1, 40_000])
@pytest.mark.parametrize("T,C", [(1, 1), (50, 7), (2000, 300), (1 << 20, 1 << 20)])
def test_small_clouds(gpu_lib, n, T, C):
    check(gpu_lib, synth.lidar(n, 5 + n % 7), 5, 5, 15, T, C)


@pytest.mark.parametrize("n", [1 << 21, (1 << 21) + 1])
@pytest.mark.parametrize("g,T,C", [(6, 20_000, 2_000), (7, 400, 400), (3, 1 << 22, 1 << 22), (4, 1 << 21, 300)])
def test_large_clouds(gpu_lib, n, g, T, C):
    check(gpu_lib, synth.lidar(n, 9), g, 7, 12, T, C)
