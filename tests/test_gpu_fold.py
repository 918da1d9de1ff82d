"""Tiles of several bands (rows narrower than a thread's words): volumes and
images around the widths and heights where bands are folded, in every launch
shape that folds, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,H,W,r", [(4, 64, 70, (3, 4, 2)), (3, 97, 128, (4, 2, 1)), (5, 33, 65, (2, 3, 4)),
                                     (2, 128, 100, (5, 5, 1)), (3, 70, 96, (3, 3, 2)), (3, 130, 129, (2, 2, 2))])
def test_volumes(gpu_lib, D, H, W, r):
    vol = synth.boolean_spheres(D, H, W, 1.9, 5 * D * H * W // 200, seed=W)
    p = gpu_lib.lpf_build_paths_3d(*r)
    got = gpu_lib.lpf_full_3d(torch.from_numpy(vol).cuda(), p).cpu().numpy()
    assert gpu_lib.lpf_paths_status(p) == 0
    np.testing.assert_array_equal(got, oracle.lpf_full3(vol, *r))


@pytest.mark.parametrize("H,W,rx,ry", [(64, 64, 9, 10), (128, 32, 5, 20), (130, 60, 30, 12), (200, 33, 20, 64), (128, 96, 70, 20),
                                       (97, 128, 12, 64)])
def test_images(gpu_lib, H, W, rx, ry):
    img = synth.ellipses(H, W, 0.4, seed=H, axes=(3.0, 6.0))
    ref = oracle.lpf_full(img, rx, ry)
    p = gpu_lib.lpf_build_paths(rx, ry)
    d = torch.from_numpy(img).cuda()
    ran = 0
    for BB in (1, 2, 3, 4, 6, 8):
        try:
            gpu_lib.lpf_set_launch_shape(p, H, W, 8, BB)
        except gpu_lib.LpfError:
            continue
        np.testing.assert_array_equal(gpu_lib.lpf_full(d, p).cpu().numpy(), ref, err_msg=f"BB={BB}")
        ran += 1
    assert ran >= 2 and gpu_lib.lpf_paths_status(p) == 0
