"""Where the group passes of fp_build_ooc keep things: a second set of group
buffers, the whole cloud's codes and the staged points fit the dead piece buffers
or not (pieces from large to small), staged points come back in bulk or are read
one by one (arenas down to a few groups' worth), one group and many, an odd and an
even number of them.  Exactly the in-core build's outputs in every case."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

N = 16_000_000


@pytest.fixture(scope="module")
def cloud(gpu_lib):
    fp = gpu_lib
    dev = fp.as_points(synth.uniform(N, 46), "cuda")
    return dev, dev.cpu().pin_memory()


@pytest.mark.parametrize("piece,group,T,less", [
    (1 << 21, 0, 300_000, 0), (1 << 19, 0, 300_000, 0), (1 << 17, 0, 300_000, 0),
    (1 << 21, 0, 100_000, 0), (1 << 19, 0, 100_000, 0), (1 << 19, 0, 100_000, 30 << 20),
    (1 << 19, 260_000, 300_000, 0), (1 << 21, 260_000, 300_000, 0), (1 << 17, 270_000, 300_000, 60 << 20)])
def test_groups(gpu_lib, cloud, piece, group, T, less):
    fp = gpu_lib
    dev, host = cloud
    prm = fp.params(5, 5, 12, 16, T, 20_000)
    ref = fp.build_octree(dev, prm)
    arena = torch.empty(fp.ooc_arena_min(N, prm, piece) - less, dtype=torch.uint8, device="cuda")
    out = fp.build_ooc(host, prm, arena, piece_points=piece, group_points=group)
    assert fp.get_device_error() == 0
    M = int(ref["num_nodes"].item())
    assert int(out["num_nodes"].item()) == M
    rows = lambda t: t[:M].cpu().contiguous().view(torch.uint8).reshape(M, 40)
    assert torch.equal(rows(out["nodes"]), rows(ref["nodes"]))
    assert torch.equal(out["final_perm"][:N], ref["final_perm"].cpu())
    assert torch.equal(out["final"][:N], ref["final"].cpu())
