"""The uniform preview without extents on each of its paths (two launches with
small tiles; one cooperative launch from 608 tiles of 8192 points on; two launches
with large tiles beyond 24 tiles a block) and its keep rule at moduli of every
kind (powers of two, odd, mixed, the extremes), against the oracle, or for the
largest piece against the pass with extents.  Whole numbers: no tolerance."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import assert_points_equal, dev_points

pytestmark = pytest.mark.gpu

EDGE = 608 * 8192   # first size of the cooperative path on 152 SMs


@pytest.fixture(scope="module")
def cloud():
    pts = synth.uniform(EDGE + 8193, 71)
    return pts, dev_points(pts)


@pytest.mark.parametrize("n", [1, 2047, 2049, EDGE - 8192, EDGE - 8191, EDGE, EDGE + 1, EDGE + 8193])
@pytest.mark.parametrize("modulus,first", [(16, 0), (52, (1 << 40) + 3)])
def test_decimate_sizes(gpu_lib, cloud, n, modulus, first):
    fp, (pts_np, pts) = gpu_lib, cloud
    out, count = fp.fp_decimate(pts[:n], first, modulus)
    want = oracle.decimate(pts_np[:n], first, modulus)[0]
    assert fp.get_device_error() == 0
    assert int(count.item()) == len(want)
    assert_points_equal(out, want, count=len(want))


@pytest.mark.parametrize("modulus", [1, 2, 3, 7, 12, 96, 1000003, 3 << 30, 1 << 31, (1 << 32) - 1])
def test_keep_rule(gpu_lib, cloud, modulus):
    fp, (pts_np, pts) = gpu_lib, cloud
    n = 300_001
    want = oracle.decimate(pts_np[:n], 5, modulus)[0]
    out, count = fp.fp_decimate(pts[:n], 5, modulus)
    assert int(count.item()) == len(want)
    assert_points_equal(out, want, count=len(want))
    _, out, count = fp.fp_bounds_decimate(pts[:n], 5, modulus)
    assert int(count.item()) == len(want)
    assert_points_equal(out, want, count=len(want))


def test_decimate_capacity(gpu_lib, cloud):
    fp, (pts_np, pts) = gpu_lib, cloud
    fp.get_device_error(clear=True)
    want = oracle.decimate(pts_np, 0, 16)[0]
    out = torch.zeros((1000, 4), dtype=torch.int32, device="cuda")
    _, count = fp.fp_decimate(pts, 0, 16, out=out[:900])
    assert int(count.item()) == len(want)
    assert fp.get_device_error() & (1 << 9)
    assert_points_equal(out, want[:900], count=900)
    assert int(out[900:].abs().sum().item()) == 0


def test_decimate_beyond_the_cooperative_path(gpu_lib):
    fp = gpu_lib
    n = 152 * 8 * 24 * 8192 + 1
    pts = torch.arange(4 * n, dtype=torch.int32, device="cuda").view(n, 4)
    a, ca = fp.fp_decimate(pts, 9, 1000)
    _, b, cb = fp.fp_bounds_decimate(pts, 9, 1000)
    assert fp.get_device_error() == 0
    k = int(ca.item())
    assert k == int(cb.item()) and torch.equal(a[:k], b[:k])


# around the tile of 8192 points; grids of 8 cells and of 2^21; LiDAR's empty cells
@pytest.mark.parametrize("n", [1, 31, 33, 8191, 8192, 8193, 100_003])
@pytest.mark.parametrize("level", [1, 4, 7])
def test_spatial_sizes(gpu_lib, n, level):
    fp = gpu_lib
    pts_np = synth.lidar(n, 72)
    cube, pts = oracle.bounds(pts_np), dev_points(pts_np)
    out, count = fp.fp_preview_spatial(pts, fp.fp_bounds(pts), level, (1 << 33) + n)
    want, _ = oracle.preview_spatial(pts_np, cube, level, (1 << 33) + n)
    assert int(count.item()) == len(want)
    assert_points_equal(out, want, count=len(want))


# the one index whose hash is the largest value (it marks empty cells on the device): alone in its cell, or not
@pytest.mark.parametrize("alone", [False, True])
def test_spatial_largest_hash(gpu_lib, alone):
    fp = gpu_lib
    first = (0x31628AF67B2131AB - 5) % (1 << 64)
    pts_np = synth.uniform(64, 73, bits=10)
    pts_np["x"][5] = 4000 if alone else pts_np["x"][6]
    if not alone:
        pts_np["y"][5], pts_np["z"][5] = pts_np["y"][6], pts_np["z"][6]
    pts = dev_points(pts_np)
    out, count = fp.fp_preview_spatial(pts, fp.fp_bounds(pts), 3, first)
    want, _ = oracle.preview_spatial(pts_np, oracle.bounds(pts_np), 3, first)
    assert int(count.item()) == len(want)
    assert_points_equal(out, want, count=len(want))
