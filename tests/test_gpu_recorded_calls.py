"""Calls recorded into a CUDA graph: they stay valid while the same handle
evaluates ensembles (their work areas do not move), and after one plain
evaluation of an image its ensembles can be recorded, and the other way
round."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


def _graph(call):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    return g


def _images(n, H, W, seed):
    return np.stack([synth.random_binary(H, W, 0.6, seed + k) for k in range(n)])


def test_recorded_evaluations_outlive_larger_ensembles(gpu_lib):
    H, W, rx, ry = 40, 61, 13, 9
    first, few, many = _images(1, H, W, 1), _images(4, H, W, 10), _images(200, H, W, 40)
    ref = {id(a): sum(oracle.lpf_full(i, rx, ry) for i in a) for a in (first, few, many)}
    p = gpu_lib.lpf_build_paths(rx, ry)
    d1, d4, d200 = (torch.from_numpy(a).cuda() for a in (first, few, many))
    c1, c4 = (torch.empty((2, p.n_full), dtype=torch.int64, device="cuda") for _ in range(2))
    gpu_lib.lpf_full(d1[0], p, c1)
    gpu_lib.lpf_full_ensemble(d4, p, c4)
    g1 = _graph(lambda: gpu_lib.lpf_full(d1[0], p, c1))
    g4 = _graph(lambda: gpu_lib.lpf_full_ensemble(d4, p, c4))
    np.testing.assert_array_equal(gpu_lib.lpf_full_ensemble(d200, p).cpu().numpy(), ref[id(many)])
    scratch = torch.full((64 << 18,), -1, dtype=torch.int32, device="cuda")  # what the allocator hands out next
    c1.zero_(), c4.zero_()
    g1.replay(), g4.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(c1.cpu().numpy(), ref[id(first)])
    np.testing.assert_array_equal(c4.cpu().numpy(), ref[id(few)])
    assert (scratch == -1).all() and gpu_lib.lpf_paths_status(p) == 0


def test_recorded_ensemble_after_a_plain_evaluation(gpu_lib):
    H, W, rx, ry = 40, 61, 13, 9
    imgs = _images(5, H, W, 7)
    p = gpu_lib.lpf_build_paths(rx, ry)
    d, c = torch.from_numpy(imgs).cuda(), torch.empty((2, p.n_full), dtype=torch.int64, device="cuda")
    gpu_lib.lpf_full(d[0], p)
    _graph(lambda: gpu_lib.lpf_full_ensemble(d, p, c)).replay()
    np.testing.assert_array_equal(c.cpu().numpy(), sum(oracle.lpf_full(i, rx, ry) for i in imgs))
    gpu_lib.lpf_full_ensemble(d[:3].contiguous(), p)  # now an area for three, still none for five
    c.zero_()
    _graph(lambda: gpu_lib.lpf_full_ensemble(d, p, c)).replay()
    np.testing.assert_array_equal(c.cpu().numpy(), sum(oracle.lpf_full(i, rx, ry) for i in imgs))


def test_recorded_evaluation_after_a_plain_ensemble(gpu_lib):
    H, W, rx, ry = 40, 61, 30, 28
    imgs = _images(200, H, W, 7)  # enough for the long pieces, which one image would not take
    p = gpu_lib.lpf_build_paths(rx, ry)
    d, c = torch.from_numpy(imgs).cuda(), torch.empty((2, p.n_full), dtype=torch.int64, device="cuda")
    gpu_lib.lpf_full_ensemble(d, p)
    _graph(lambda: gpu_lib.lpf_full(d[0], p, c)).replay()
    np.testing.assert_array_equal(c.cpu().numpy(), oracle.lpf_full(imgs[0], rx, ry))
    assert gpu_lib.lpf_paths_status(p) == 0
