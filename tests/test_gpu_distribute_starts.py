"""fp_distribute puts point r of chunk c at d_offsets[c] + r, whatever the order of the
starts: chunks in reverse and in random order, on both sides of the size where the
distribution changes from one cluster to the sweeps, with the cells given and not; and
starts that reach beyond the output (reported; everything else is placed)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import dev_points, host_points

pytestmark = pytest.mark.gpu

G = 5
SITE = 15   # a position beyond the output


def expected(cells, lut, starts):
    """Output position of every point."""
    c = lut[cells]
    order = np.argsort(c, kind="stable")
    first = np.searchsorted(c[order], np.arange(len(starts)))
    pos = np.empty(len(c), np.int64)
    pos[order] = starts[c[order]] + np.arange(len(c)) - first[c[order]]
    return pos


@pytest.mark.parametrize("n", [1, 1000, (1 << 15) - 1, 1 << 15, (1 << 15) + 1, 50_003])
@pytest.mark.parametrize("K", [1, 2, 300, 1500])
@pytest.mark.parametrize("order", ["reverse", "random", "shifted"])
def test_chunk_starts_in_any_order(gpu_lib, n, K, order):
    fp = gpu_lib
    pts = synth.uniform(n, 97)
    cube = oracle.bounds(pts)
    cells = oracle.point_keys(pts, cube, G).astype(np.int64)
    lut = (np.arange(1 << (3 * G)) * K >> (3 * G)).astype(np.int64)
    count = np.bincount(lut[cells], minlength=K)
    seq = np.arange(K)[::-1] if order == "reverse" else np.random.default_rng(n).permutation(K)
    starts = np.empty(K, np.int64)
    starts[seq] = np.cumsum(count[seq]) - count[seq]
    if order == "shifted":
        starts = np.cumsum(count) - count + 7
    pos = expected(cells, lut, starts)
    dev = dev_points(pts)
    dcube = fp.fp_bounds(dev)
    t = lambda a, d: torch.from_numpy(np.ascontiguousarray(a)).to(d).cuda()   # noqa: E731
    off, num = t(np.append(starts, n), torch.int64), t(np.array([K]), torch.int32)
    for given in (True, False):
        fp.get_device_error(clear=True)
        out = torch.zeros((n, 4), dtype=torch.int32, device="cuda")
        perm = torch.zeros(n, dtype=torch.int32, device="cuda")
        args = (dcube, G, t(lut, torch.int32), off, num)
        if given:
            fp.fp_distribute_cells(dev, t(cells, torch.int32), *args, out=out, perm=perm)
        else:
            fp.fp_distribute(dev, *args, out=out, perm=perm)
        torch.cuda.synchronize()
        sites = fp.get_device_error_sites()
        assert bool(fp.get_device_error(clear=True) & (1 << 9)) == bool((pos >= n).any())
        assert sites == ((1 << SITE) if (pos >= n).any() else 0)
        inside = np.flatnonzero(pos < n)
        assert np.array_equal(perm.cpu().numpy()[pos[inside]], inside)
        assert np.array_equal(host_points(out)[pos[inside]], pts[inside])
