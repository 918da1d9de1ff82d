"""A volume's evaluation takes no longer than in a plain shape (one word per
thread, four bands per band group) with windows of 128 and more, whose walk does
not re-deal masks (bound: a sixth over)."""
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


@pytest.mark.parametrize("D,H,W,rx,ry,rz,T", [(3, 160, 50, 2, 130, 1, 1)])
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
