"""Volumes with nearly as many band groups as the walk has counters for: heights
of an odd number of pairs of bands, which are grouped by two where that many
groups fit and by four beyond."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,H,W", [(2730, 161, 65), (2731, 161, 65), (4000, 192, 70)])
def test_counts_of_neighbours(gpu_lib, D, H, W):
    g = torch.Generator(device="cuda").manual_seed(D)
    vol = (torch.rand((D, H, W), generator=g, device="cuda") < 0.4).to(torch.uint8)
    p = gpu_lib.lpf_build_paths_3d(1, 1, 1)
    got = gpu_lib.lpf_full_3d(vol, p).cpu()
    assert gpu_lib.lpf_paths_status(p) == 0
    for k in range(14):  # (the segment to a neighbour is its two ends)
        dz, dy, dx = k // 9 - 1, k // 3 % 3 - 1, k % 3 - 1
        both = vol + torch.roll(vol, (-dz, -dy, -dx), (0, 1, 2))
        n0, n1 = int((both == 0).sum()), int((both == 2).sum())
        assert (got[0, k], got[1, k]) == (n0, n1) and (got[0, 26 - k], got[1, 26 - k]) == (n0, n1)
