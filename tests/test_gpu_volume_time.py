"""A volume's evaluation takes no longer than in a plain shape (one band per
tile, four per band group), whatever shape is chosen for it: windows of 128 and
more, of a few pixels, and those that fold bands gain from (bound: a sixth
over)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _us(call, n=10):
    call()
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    best = float("inf")
    for _ in range(5):
        torch.cuda.synchronize()
        a.record()
        for _ in range(n):
            call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / n * 1e3)
    return best


@pytest.mark.parametrize("D,H,W,rx,ry,rz,T", [
    (3, 160, 50, 2, 130, 1, 1),
    (3, 192, 100, 2, 130, 1, 4), (3, 256, 70, 2, 130, 1, 4),
    (100, 320, 128, 4, 4, 4, 4), (128, 192, 128, 4, 4, 4, 4), (200, 192, 100, 6, 6, 6, 4), (128, 128, 128, 4, 4, 4, 4),
    (64, 128, 128, 8, 8, 8, 4), (100, 320, 128, 10, 10, 10, 4),
])
def test_no_longer_than_the_plain_shape(gpu_lib, D, H, W, rx, ry, rz, T):
    g = torch.Generator(device="cuda").manual_seed(D)
    blocks = torch.rand((D // 8 + 1, H // 8 + 1, W // 8 + 1), generator=g, device="cuda") < 0.4
    for axis in range(3):
        blocks = blocks.repeat_interleave(8, axis)
    vol = blocks[:D, :H, :W].contiguous().to(torch.uint8)
    chosen, plain = (gpu_lib.lpf_build_paths_3d(rx, ry, rz) for _ in range(2))
    gpu_lib.lpf_set_launch_shape(plain, H, W, T, min(4, -(-H // 32)))
    counts = [torch.empty((2, p.n_full), dtype=torch.int64, device="cuda") for p in (chosen, plain)]
    us = [_us(lambda: gpu_lib.lpf_full_3d(vol, p, c)) for p, c in zip((chosen, plain), counts)]
    assert torch.equal(*counts)
    assert us[0] <= 7 / 6 * us[1], us


@pytest.mark.parametrize("D,H,W,r", [(64, 64, 100, 8), (16, 128, 70, 10), (12, 192, 128, 9), (20, 128, 97, 9)])
def test_folded_tiles_count_the_same(gpu_lib, D, H, W, r):
    g = torch.Generator(device="cuda").manual_seed(D)
    vol = (torch.rand((D, H, W), generator=g, device="cuda") < 0.7).to(torch.uint8)
    chosen, plain = (gpu_lib.lpf_build_paths_3d(r, r, r) for _ in range(2))
    gpu_lib.lpf_set_launch_shape(plain, H, W, 1, 1)
    assert torch.equal(gpu_lib.lpf_full_3d(vol, chosen), gpu_lib.lpf_full_3d(vol, plain))
    assert gpu_lib.lpf_paths_status(chosen) == 0 and gpu_lib.lpf_paths_status(plain) == 0
