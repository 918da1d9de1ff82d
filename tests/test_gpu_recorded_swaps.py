"""Count changes recorded into a CUDA graph stay valid after calls with more
candidates on the same handle, whose work area is larger."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [5, 40])  # looked up one by one; from sums for every pixel
def test_recorded_count_changes_outlive_larger_calls(gpu_lib, K):
    H, W, rx, ry = 40, 61, 9, 7
    cells = [synth.random_binary(H, W, 0.4, seed=k) for k in (1, 2)]
    pairs = synth.swap_candidates(cells[0], K, seed=3).astype(np.int32)
    p = gpu_lib.lpf_build_paths(rx, ry)
    d, t = torch.from_numpy(cells[0]).cuda(), torch.from_numpy(pairs).cuda()
    dc = torch.empty((K, 2, oracle.window_sizes(rx, ry)[1]), dtype=torch.int32, device="cuda")
    gpu_lib.lpf_delta_swap(d, p, t, dcounts=dc)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        gpu_lib.lpf_delta_swap(d, p, t, dcounts=dc)
    for more in (300, 5000):
        gpu_lib.lpf_delta_swap(d, p, torch.from_numpy(synth.swap_candidates(cells[0], more, seed=4).astype(np.int32)).cuda())
    scratch = torch.full((1 << 20,), -1, dtype=torch.int32, device="cuda")  # what the allocator hands out next
    for cell in cells[::-1]:
        d.copy_(torch.from_numpy(cell))
        dc.zero_()
        g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(dc.cpu().numpy(), oracle.delta_swap(cell, rx, ry, pairs))
    assert (scratch == -1).all() and gpu_lib.lpf_paths_status(p) == 0
