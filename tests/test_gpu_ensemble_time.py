"""Images evaluated side by side take no longer than one after another, also
where one of them alone fills the GPU (bound: a quarter over; they took up to
half as long again while an SM's blocks ran two copies of the walk)."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _us(call, n=10):
    call()
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    best = float("inf")
    for _ in range(3):
        torch.cuda.synchronize()
        a.record()
        for _ in range(n):
            call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / n * 1e3)
    return best


@pytest.mark.parametrize("n,H,W,r", [(5, 239, 230, 119), (8, 128, 256, 100), (4, 256, 256, 140)])
def test_no_longer_than_one_by_one(gpu_lib, n, H, W, r):
    imgs = torch.stack([torch.from_numpy(synth.squares(H, W, 12, 0.3, seed=k)) for k in range(n)]).cuda()
    p = gpu_lib.lpf_build_paths(r, min(r, H - 1))
    counts = torch.empty((2, p.n_full), dtype=torch.int64, device="cuda")
    together = _us(lambda: gpu_lib.lpf_full_ensemble(imgs, p, counts))
    alone = _us(lambda: [gpu_lib.lpf_full(i, p, counts) for i in imgs])
    assert together <= 1.25 * alone, (together, alone)
