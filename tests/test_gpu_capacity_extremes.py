"""Node capacities and chunk thresholds at the ends of their 64-bit range: a tree of
one node, as "never split" is written, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import assert_build_matches_oracle, assert_points_equal, dev_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 5_000, 40_000])
@pytest.mark.parametrize("T,C", [((1 << 64) - 1, (1 << 64) - 1), ((1 << 64) - 1, 300), ((1 << 32) - 1, (1 << 32) - 1),
                                 (1 << 32, 1 << 32), ((1 << 63) + 5, 5_000), ((1 << 32) + 7, 4_999)])
def test_extreme_capacities(gpu_lib, n, T, C):
    fp = gpu_lib
    pts = synth.uniform(n, 98)
    r = fp.build_octree(dev_points(pts), fp.params(5, 6, 12, 16, T, C))
    torch.cuda.synchronize()
    assert fp.get_device_error() == 0
    want = oracle.build_all(pts, oracle.params(5, 6, 12, 16, T, C))
    M = int(r["num_nodes"].item())
    assert_build_matches_oracle(want, cube=r["cube"], nodes=r["nodes"][:M], final=r["final"],
                                final_perm=r["final_perm"])
    assert np.array_equal(r["leaf_perm"].cpu().numpy().view(np.uint32), want["leaf_perm"])
    assert_points_equal(r["leaf_pts"], want["leaf_pts"])
