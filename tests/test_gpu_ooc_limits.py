"""Out-of-core builds in arenas that are just large enough: the smallest ones that took
these clouds before the sorts had a second set of look-back words (the largest chunk
and the sort of the staged points set the limit), with groups as large as the arena
allows and smaller ones, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import assert_build_matches_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,g,T,C,piece,group,arena", [
    (1_000_000, 3, 130_000, 20_000, 1 << 16, 0, 30_072_832), (1_000_000, 3, 130_000, 20_000, 1 << 16, 200_000, 30_072_832),
    (1_000_000, 3, 130_000, 20_000, 1 << 14, 0, 27_451_392), (1_000_000, 3, 20_000, 2_000, 1 << 16, 0, 39_068_160),
    (500_000, 3, 10_000, 1_000, 1 << 12, 0, 20_361_216), (3_000_000, 5, 50_000, 5_000, 1 << 16, 0, 101_964_800),
    (3_000_000, 2, 400_000, 5_000, 1 << 17, 0, 63_815_680)])
def test_smallest_arenas(gpu_lib, n, g, T, C, piece, group, arena):
    fp = gpu_lib
    pts = synth.uniform(n, 5)
    prm = (g, 7, 12, 16, T, C)
    host = torch.from_numpy(pts.view(np.int32).reshape(-1, 4)).pin_memory()
    out = fp.build_ooc(host, fp.params(*prm), torch.empty(arena, dtype=torch.uint8, device="cuda"), piece_points=piece,
                       group_points=group)
    assert fp.get_device_error() == 0
    M = int(out["num_nodes"][0])
    assert_build_matches_oracle(oracle.build_all(pts, oracle.params(*prm)), cube=out["cube"], preview=out["preview"],
                                nodes=out["nodes"][:M], final=out["final"], final_perm=out["final_perm"])
