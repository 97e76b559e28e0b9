"""Device memory the calls ask for: callers size buffers and arenas once, so what was
enough before a change of the kernels has to be enough after it.  The limits are the
sizes of the library before its sorts and the distribution got a second set of tables."""

import pytest

from paper_2302_05002_gb300 import fastpoints as fp


@pytest.mark.parametrize("n,most", [(1_000, 146_176), (20_000, 595_712), (200_000, 4_961_792), (1_000_000, 24_424_448),
                                    (5_000_000, 121_684_736), (30_000_000, 729_548_288), (300_000_000, 7_294_451_712)])
def test_distribution_workspace(n, most):
    assert fp.workspace_size("distribute", n, fp.params(grid_log2=7)) <= most


@pytest.mark.parametrize("n,g,C,lmax,piece,most", [
    (1, 1, 50, 15, 1 << 21, 162_827_008), (20_000, 7, 20_000, 15, 1 << 12, 808_697_344),
    (1_000_000, 3, 50, 12, 1 << 16, 403_309_568), (1_000_000, 5, 1, 12, 1 << 12, 482_033_408),
    (5_000_000, 7, 20_000, 15, 1 << 21, 1_040_546_560), (30_000_000, 7, 20_000, 15, 1 << 23, 1_382_548_480),
    (300_000_000, 7, 50, 12, 1 << 23, 39_365_628_928), (300_000_000, 1, 50, 15, 1 << 12, 80_013_739_264)])
def test_smallest_arena(n, g, C, lmax, piece, most):
    assert fp.ooc_arena_min(n, fp.params(g, 7, lmax, 16, max(C, 100_000), C), piece) <= most
