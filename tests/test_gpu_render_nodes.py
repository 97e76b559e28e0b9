"""Frames of trees with many small nodes: drawn nodes without points (more than a
thousand of them between two points of a run), nodes of one point, of a few, against
the oracle bit by bit; and such a frame is not several times that of a coarse tree."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import dev_points
from tests.test_gpu_render import cameras

pytestmark = pytest.mark.gpu


# the root keeps nearly every point (2^12 cells an axis), or few (2^4)
@pytest.mark.parametrize("n,s,C", [(30_000, 12, 1), (200_000, 10, 1), (200_000, 4, 2), (400_000, 7, 5)])
def test_many_nodes(gpu_lib, n, s, C):
    fp = gpu_lib
    pts_np = synth.lidar(n, 111)
    prm = fp.params(grid_log2=4, sub_log2=s, max_level=22 - s if s > 8 else 14, chunk_threshold=2000, node_capacity=C)
    r = fp.build_octree(dev_points(pts_np), prm)
    nodes_h = fp.nodes_to_host(r["nodes"], r["num_nodes"])
    cube, (W, H) = oracle.bounds(pts_np), (640, 360)
    fin = r["final"].cpu().numpy().view(np.uint8).reshape(-1, 16).copy().view(oracle.POINT).reshape(-1)
    for name, m, _ in cameras(fp, pts_np, W, H):
        cam, ocam = fp.camera(m, W, H, 0.0), oracle.camera(m, W, H, 0.0)
        ids, nsel, _ = fp.fp_select_nodes(r["nodes"], r["num_nodes"], r["cube"], cam)
        fb = fp.fp_rasterize(r["nodes"], ids, nsel, r["final"], cam)
        torch.cuda.synchronize()
        assert fp.get_device_error() == 0
        sel = ids[:int(nsel.item())].cpu().numpy().view(np.uint32)
        assert np.array_equal(sel, oracle.render_select(nodes_h, cube, ocam)), name
        assert np.array_equal(fb.cpu().numpy().view(np.uint64).reshape(-1),
                              oracle.rasterize(nodes_h, sel, fin, ocam).reshape(-1)), name


def test_small_nodes_are_no_search(gpu_lib):
    fp, n, ms = gpu_lib, 3_000_000, []
    pts = torch.randint(0, 1 << 20, (n, 4), dtype=torch.int32, device="cuda")
    for k in range(2):
        pts[:, k] = (torch.rand(n, device="cuda") ** 2 * (1 << 20)).to(torch.int32)
    pts[:, 2] //= 16
    cam = fp.camera(fp.view_projection([5e5, -4e5, 6e5], [5e5, 5e5, 0.0], aspect=16 / 9, near=1.0, far=4e6), 3840, 2160, 2.0)
    fb = torch.empty((2160, 3840), dtype=torch.int64, device="cuda")
    for C in (20_000, 40):
        r = fp.build_octree(pts, fp.params(7, 7, 14, 16, 20_000, C))
        nodes = r["nodes"][:int(r["num_nodes"].item())].contiguous()
        ws = torch.empty(fp.render_workspace_size(nodes.shape[0]), dtype=torch.uint8, device="cuda")
        ids, nsel, npts = fp.fp_select_nodes(nodes, r["num_nodes"], r["cube"], cam, ws=ws)
        one = []
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            fp.fp_rasterize(nodes, ids, nsel, r["final"], cam, fb=fb, ws=ws)
            b.record()
            b.synchronize()
            one.append(a.elapsed_time(b))
        ms.append((sorted(one)[4], int(nsel.item()), int(npts.item())))
    assert fp.get_device_error() == 0
    assert ms[1][0] < 1.5 * ms[0][0], ms
