"""The renderer's two launches at the sizes where their split changes: fewer nodes
than blocks, more nodes than a block's share of one round, drawn nodes of one
point each (every warp's run crosses nodes), one node with all points,
framebuffers of one pixel, odd widths, and a node table with room behind it.
Everything against the oracle, bit by bit."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import dev_points
from tests.test_gpu_render import cameras

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,C,W,H", [(2, 1, 1, 1), (3, 1, 1, 7), (127, 1 << 20, 5, 3), (129, 1, 33, 17),
                                     (60_000, 1, 257, 129), (60_000, 1 << 20, 64, 48), (700_000, 40, 1001, 333)])
@pytest.mark.parametrize("minpx", [0.0, 3.0])
def test_runs(gpu_lib, n, C, W, H, minpx):
    fp = gpu_lib
    pts_np = synth.lidar(n, 90 + n % 9)
    prm = fp.params(grid_log2=5, sub_log2=5, max_level=14, chunk_threshold=max(C, 2000), node_capacity=C)
    r = fp.build_octree(dev_points(pts_np), prm)
    nodes_h = fp.nodes_to_host(r["nodes"], r["num_nodes"])
    cube = oracle.bounds(pts_np)
    fin = r["final"].cpu().numpy().view(np.uint8).reshape(-1, 16).copy().view(oracle.POINT).reshape(-1)
    for name, m, _ in cameras(fp, pts_np, W, H):
        cam, ocam = fp.camera(m, W, H, minpx), oracle.camera(m, W, H, minpx)
        want_sel = oracle.render_select(nodes_h, cube, ocam)
        ids, nsel, npts = fp.fp_select_nodes(r["nodes"], r["num_nodes"], r["cube"], cam)
        fb = fp.fp_rasterize(r["nodes"], ids, nsel, r["final"], cam)
        torch.cuda.synchronize()
        assert fp.get_device_error() == 0
        k = int(nsel.item())
        assert np.array_equal(ids[:k].cpu().numpy().view(np.uint32), want_sel), name
        assert int(npts.item()) == int(nodes_h["n_own"][want_sel].astype(np.int64).sum())
        want_fb = oracle.rasterize(nodes_h, want_sel, fin, ocam).reshape(-1)
        assert np.array_equal(fb.cpu().numpy().view(np.uint64).reshape(-1), want_fb), name
