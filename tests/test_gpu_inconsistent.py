"""Inputs that contradict each other end in FP_ERR_CAPACITY with every access inside
the buffers, and the call after them is right again."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import assert_build_matches_oracle, dev_points

pytestmark = pytest.mark.gpu

CAPACITY = 1 << 9


def rebuild(fp, pts, prm):
    r = fp.build_octree(dev_points(pts), fp.params(*prm))
    torch.cuda.synchronize()
    assert fp.get_device_error() == 0
    want = oracle.build_all(pts, oracle.params(*prm))
    M = int(r["num_nodes"].item())
    assert_build_matches_oracle(want, nodes=r["nodes"][:M], final=r["final"], final_perm=r["final_perm"])


@pytest.mark.parametrize("g", [1, 2, 5, 7])
@pytest.mark.parametrize("n", [900, 30_000, 600_000])
@pytest.mark.parametrize("wrong", ["none", "other", "one", "more"])
def test_a_count_grid_of_other_points(gpu_lib, g, n, wrong):
    """Points that no piece holds have no code; whatever their word held before, the
    owner search stays in its tables (workspace filled with ones)."""
    fp = gpu_lib
    prm = (g, 7, 12, 16, 5_000, 500)
    pts = synth.uniform(n, 103)
    dev, p = dev_points(pts), fp.params(*prm)
    cube = fp.fp_bounds(dev)
    counts = fp.fp_count(dev, cube, g)
    chunks, num, lut, offsets = fp.fp_merge_chunks(counts, g, prm[4])
    dist, perm = fp.fp_distribute(dev, cube, g, lut, offsets, num)
    if wrong == "none":
        bad = torch.zeros_like(counts)
    elif wrong == "other":
        bad = counts.flip(0).contiguous()
        bad[0] += 1
    elif wrong == "one":
        bad = torch.zeros_like(counts)
        bad[3] = n
    else:
        bad = counts * 2 + 1
    ws = torch.full((fp.workspace_size("octree", n, p),), 255, dtype=torch.uint8, device="cuda")
    fp.get_device_error(clear=True)
    fp.fp_build_chunk_octree(dist, perm, cube, chunks, num, offsets, bad, p, leaf=True, ws=ws)
    torch.cuda.synchronize()
    assert fp.get_device_error(clear=True) & CAPACITY
    rebuild(fp, synth.uniform(5_000, 104), prm)


def test_more_owned_points_than_points(gpu_lib):
    """A node table whose owned counts add up to 2^32 and more (not the table of these points)."""
    fp = gpu_lib
    n, prm = (1 << 21) + 5_000, (7, 7, 12, 16, 50_000, 5_000)
    dev, p = dev_points(synth.uniform(n, 105)), fp.params(*prm)
    cube = fp.fp_bounds(dev)
    counts = fp.fp_count(dev, cube, 7)
    chunks, num, lut, offsets = fp.fp_merge_chunks(counts, 7, prm[4])
    dist, perm = fp.fp_distribute(dev, cube, 7, lut, offsets, num)
    nodes, m, _, _, owner = fp.fp_build_chunk_octree(dist, perm, cube, chunks, num, offsets, counts, p, leaf=False)
    torch.cuda.synchronize()
    assert fp.get_device_error() == 0
    words = nodes.view(torch.int32).view(-1, 10)   # n_own is the word behind count
    M = int(m.item())
    assert int(words[:M, 7].sum().item()) == n
    words[:M:3, 7] = -1
    fp.fp_subsample(nodes, m, dist, perm, owner, chunks, num, offsets, p)
    torch.cuda.synchronize()
    assert fp.get_device_error(clear=True) & CAPACITY
    rebuild(fp, synth.uniform(5_000, 106), prm)
