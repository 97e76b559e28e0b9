"""Device memory the calls ask for: callers size buffers and arenas once, so what was
enough before a change of the kernels has to be enough after it.  The limits are the
sizes of the library before its sorts and the distribution got a second set of tables."""

import pytest

from paper_2302_05002_gb300 import fastpoints as fp


@pytest.mark.parametrize("n,most", [(1_000, 146_176), (20_000, 595_712), (200_000, 4_961_792), (1_000_000, 24_424_448),
                                    (5_000_000, 121_684_736), (30_000_000, 729_548_288), (300_000_000, 7_294_451_712)])
def test_distribution_workspace(n, most):
    assert fp.workspace_size("distribute", n, fp.params(grid_log2=7)) <= most
