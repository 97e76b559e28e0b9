"""The chunk-wise layouts (clouds of more than 2^21 points) with chunks of very unequal
sizes: all points in one chunk, one chunk of nearly all points among thousands, and
chunks of a tile more or less; the final layout and the leaf grouping against the
oracle.  And one chunk's look-back words are cleared by every warp."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import assert_build_matches_oracle, assert_points_equal, dev_points

pytestmark = pytest.mark.gpu

N = (1 << 21) + 70_003


def cloud(kind):
    pts = synth.uniform(N, 101)
    if kind == "crowded":   # nine points in ten in one level-5 cell
        hot = np.random.default_rng(4).random(N) < 0.9
        for a in "xyz":
            pts[a][hot] = (3 << 15) + pts[a][hot] % (1 << 15)
    return pts


@pytest.mark.parametrize("kind,g,T,C", [("even", 5, 60, 60), ("crowded", 1, 1 << 40, 20_000), ("crowded", 5, 1 << 40, 20_000),
                                        ("crowded", 5, 4_096, 4_096), ("crowded", 3, 300_000, 9_000)])
def test_unequal_chunks(gpu_lib, kind, g, T, C):
    fp = gpu_lib
    pts = cloud(kind)
    r = fp.build_octree(dev_points(pts), fp.params(g, 5, 9, 16, T, C))
    torch.cuda.synchronize()
    assert fp.get_device_error() == 0
    want = oracle.build_all(pts, oracle.params(g, 5, 9, 16, T, C))
    M = int(r["num_nodes"].item())
    assert_build_matches_oracle(want, nodes=r["nodes"][:M], final=r["final"], final_perm=r["final_perm"])
    assert np.array_equal(r["leaf_perm"].cpu().numpy().view(np.uint32), want["leaf_perm"])
    assert_points_equal(r["leaf_pts"], want["leaf_pts"])


def median_ms(call):
    ms = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        b.synchronize()
        ms.append(a.elapsed_time(b))
    return sorted(ms)[4]


def test_one_chunk_is_no_chain(gpu_lib):
    """The final layout of a cloud that is one chunk moves little more than its
    distribution does (1.9 times as long; 4 times with one warp clearing)."""
    fp, n = gpu_lib, 30_000_000
    pts = torch.randint(0, 1 << 20, (n, 4), dtype=torch.int32, device="cuda")
    prm = fp.params(7, 7, 15, 16, 1 << 40, n // 300)
    cube = fp.fp_bounds(pts)
    counts = fp.fp_count(pts, cube, 7)
    chunks, num, lut, offsets = fp.fp_merge_chunks(counts, 7, 1 << 40)
    ws = torch.empty(max(fp.workspace_size(k, n, prm) for k in ("distribute", "octree", "subsample")),
                     dtype=torch.uint8, device="cuda")
    dist, perm = fp.fp_distribute(pts, cube, 7, lut, offsets, num, ws=ws)
    nodes, m, _, _, owner = fp.fp_build_chunk_octree(dist, perm, cube, chunks, num, offsets, counts, prm, leaf=False,
                                                     ws=ws)
    final, final_perm = torch.empty_like(pts), torch.empty_like(perm)
    distribute = median_ms(lambda: fp.fp_distribute(pts, cube, 7, lut, offsets, num, out=dist, perm=perm, ws=ws))
    layout = median_ms(lambda: fp.fp_subsample(nodes, m, dist, perm, owner, chunks, num, offsets, prm, ws=ws, final=final,
                                               final_perm=final_perm))
    assert fp.get_device_error() == 0
    assert layout < 3 * distribute, (layout, distribute)


# a node table of one segment, of a few, of all 512 and of several tiles each
@pytest.mark.parametrize("C", [1 << 21, 3_000, 100, 1])
def test_node_tables(gpu_lib, C):
    fp = gpu_lib
    pts = synth.uniform(N, 102)
    prm = (7, 7, 10, 16, max(C, 600), C)
    r = fp.build_octree(dev_points(pts), fp.params(*prm))
    torch.cuda.synchronize()
    assert fp.get_device_error() == 0
    want = oracle.build_all(pts, oracle.params(*prm))
    M = int(r["num_nodes"].item())
    assert_build_matches_oracle(want, nodes=r["nodes"][:M], final=r["final"], final_perm=r["final_perm"])


def test_many_nodes_are_no_chain(gpu_lib):
    """The chunk-wise scatter with 3.2 * 10^6 nodes against the same cloud's with 585: its
    plan reads the node table on the whole GPU (6.2 times as long; by one cluster 12.6)."""
    fp, n, ms = gpu_lib, N, []
    pts = torch.randint(0, 1 << 20, (n, 4), dtype=torch.int32, device="cuda")
    cube = fp.fp_bounds(pts)
    counts = fp.fp_count(pts, cube, 7)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for e in ev:
        e.record()
    torch.cuda.synchronize()
    for T, C in ((20_000, 20_000), (600, 1)):
        prm = fp.params(7, 7, 15, 16, T, C)
        chunks, num, lut, offsets = fp.fp_merge_chunks(counts, 7, T)
        dist, perm = fp.fp_distribute(pts, cube, 7, lut, offsets, num)
        nodes, m, _, _, owner = fp.fp_build_chunk_octree(dist, perm, cube, chunks, num, offsets, counts, prm, leaf=False)
        ws = torch.empty(fp.workspace_size("subsample", n, prm), dtype=torch.uint8, device="cuda")
        one = []
        fp.time_kernel("owner_scatter", ev[0], ev[1])
        for _ in range(9):
            fp.fp_subsample(nodes, m, dist, perm, owner, chunks, num, offsets, prm, ws=ws)
            torch.cuda.synchronize()
            one.append(ev[0].elapsed_time(ev[1]))
        fp.time_kernel(0)
        ms.append(sorted(one)[4])
    assert fp.get_device_error() == 0
    assert ms[1] < 9 * ms[0], ms
