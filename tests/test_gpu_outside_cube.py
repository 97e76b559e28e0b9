"""The spatial preview over a cube that does not hold the cloud (another cloud's, or
a part of it): the cube's cells repeat outside it, and every point belongs to one of
them.  Expected: exact integer cells in numpy, the smallest index hash of each."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import assert_points_equal, cube_np, dev_points

pytestmark = pytest.mark.gpu


def mix(v):
    with np.errstate(over="ignore"):
        z = v + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def expected(pts, cube, level, first):
    """Indices of the kept points."""
    key = np.zeros(len(pts), np.int64)
    S = int(cube["S"][0])
    for k, a in enumerate("xyz"):
        d = (pts[a].astype(np.int64) - int(cube["o"][0][k])) % (1 << 32)
        key = key << level | ((d << level) // S) % (1 << level)
    order = np.lexsort((mix(np.uint64(first) + np.arange(len(pts), dtype=np.uint64)), key))
    head = np.ones(len(pts), bool)
    head[1:] = key[order][1:] != key[order][:-1]
    return np.sort(order[head])


@pytest.mark.parametrize("n", [1, 33, 8193, 200_003])
@pytest.mark.parametrize("level", [1, 4, 7])
@pytest.mark.parametrize("part", [0.5, 0.01])
def test_spatial_outside_the_cube(gpu_lib, n, level, part):
    fp = gpu_lib
    pts = synth.uniform(n, 90 + level)
    for a in "xyz":
        pts[a] -= 1 << 19
    inner = synth.uniform(1000, 91)
    for a in "xyz":   # the middle of the cloud: points on all sides of it
        inner[a] = (inner[a] - (1 << 19)) * part
    cube = fp.fp_bounds(dev_points(inner))
    first = (1 << 40) + n
    out, count = fp.fp_preview_spatial(dev_points(pts), cube, level, first)
    torch.cuda.synchronize()
    assert fp.get_device_error() == 0
    want = expected(pts, cube_np(cube), level, first)
    assert int(count.item()) == len(want)
    assert_points_equal(out, pts[want], count=len(want))


def test_expected_is_the_oracles_inside(gpu_lib):
    pts = synth.lidar(20_000, 92)
    cube = oracle.bounds(pts)
    want, _ = oracle.preview_spatial(pts, cube, 5, 7)
    assert np.array_equal(pts[expected(pts, np.atleast_1d(cube), 5, 7)], want)


# one cluster, the sweeps, the radix passes
@pytest.mark.parametrize("n", [1000, 1 << 15, (1 << 15) + 1, 100_003])
@pytest.mark.parametrize("K", [8, 4097])
def test_distribute_outside_the_cube(gpu_lib, n, K):
    """Points of another cloud than the grid's: reported, and every read stays in the tables."""
    fp, g = gpu_lib, 5
    pts = synth.uniform(n, 95)
    inner = synth.uniform(1000, 96)
    for a in "xyz":
        inner[a] = inner[a] // 64 + (1 << 18)
    dev, cube = dev_points(pts), fp.fp_bounds(dev_points(inner))
    lut = (torch.arange(1 << (3 * g), dtype=torch.int64, device="cuda") * K >> (3 * g)).to(torch.int32)
    offsets = (torch.arange(K + 1, dtype=torch.int64, device="cuda") * n // K)
    num = torch.tensor([K], dtype=torch.int32, device="cuda")
    fp.get_device_error(clear=True)
    fp.fp_distribute(dev, cube, g, lut, offsets, num)
    torch.cuda.synchronize()
    sites = fp.get_device_error_sites()
    assert fp.get_device_error(clear=True) & (1 << 9)
    assert sites >> 19 & 1
