"""The count grid on both sides of the size from which a block keeps a table of
cells on chip: clouds whose points share cells (LiDAR scans, one cell, a handful)
and clouds whose points do not (the table is given up), with and without the cells
written, added to counts that are there.  Whole numbers, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import dev_points

pytestmark = pytest.mark.gpu

EDGE = 1 << 23


def cloud(kind, n):
    if kind == "lidar":
        return synth.lidar(n, 81)
    pts = synth.uniform(n, 82, bits=20)
    if kind == "few":
        for a in "xyz":
            pts[a] &= 0x80000
    if kind == "one":
        for a in "xyz":
            pts[a][:-1] = 5
    return pts


@pytest.mark.parametrize("kind", ["lidar", "uniform", "few", "one"])
@pytest.mark.parametrize("n", [EDGE - 1, EDGE, EDGE + 4097])
def test_count(gpu_lib, kind, n):
    fp = gpu_lib
    pts_np = cloud(kind, n)
    pts, ocube = dev_points(pts_np), oracle.bounds(pts_np)
    cube = fp.fp_bounds(pts)
    for g in (1, 5, 7):
        want = oracle.count(pts_np, ocube, g).astype(np.int64)
        got = fp.fp_count(pts, cube, g)
        assert np.array_equal(got.cpu().numpy().view(np.uint32), want)
        again, cells = fp.fp_count_cells(pts, cube, g, counts=got, accumulate=True)
        assert np.array_equal(again.cpu().numpy().view(np.uint32), 2 * want)
        assert np.array_equal(torch.bincount(cells.long(), minlength=1 << (3 * g)).cpu().numpy(), want)
    assert fp.get_device_error() == 0
