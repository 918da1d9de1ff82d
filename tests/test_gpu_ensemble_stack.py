"""Ensembles walked side by side: more images than one set of launches takes,
sizes whose packed rows do not end on a 16-byte boundary, wide windows, the
work reported for the last image."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,H,W,rx,ry", [(4200, 5, 6, 2, 3), (3, 33, 70, 69, 20), (17, 40, 31, 9, 1), (6, 100, 129, 64, 70),
                                         (9, 1, 40, 12, 0)])
def test_sum_over_the_images(gpu_lib, n, H, W, rx, ry):
    rng = np.random.default_rng(n)
    imgs = (rng.random((n, H, W)) < 0.3).astype(np.uint8)
    if H > 8:
        imgs |= np.roll(imgs, 1, 1) | np.roll(imgs, 1, 2)
    p = gpu_lib.lpf_build_paths(rx, ry)
    d = torch.from_numpy(imgs).cuda()
    got = gpu_lib.lpf_full_ensemble(d, p).cpu().numpy()
    assert gpu_lib.lpf_paths_status(p) == 0
    work = gpu_lib.lpf_paths_work(p)
    kinds, times = np.unique(imgs.reshape(n, -1), axis=0, return_counts=True)
    ref = sum(int(t) * oracle.lpf_full(k.reshape(H, W), rx, ry) for k, t in zip(kinds[:300], times[:300]))
    if len(kinds) > 300:  # the small images: the rest through the library one by one
        ref = ref + sum(int(t) * gpu_lib.lpf_full(torch.from_numpy(k.reshape(H, W).copy()).cuda(), p).cpu().numpy()
                        for k, t in zip(kinds[300:], times[300:]))
    np.testing.assert_array_equal(got, ref)
    np.testing.assert_array_equal(gpu_lib.lpf_full(d[-1].contiguous(), p).cpu().numpy(),
                                  oracle.lpf_full(imgs[-1], rx, ry))
    assert gpu_lib.lpf_paths_work(p) == work


def test_checked_mode_sees_every_image(gpu_lib):
    imgs = torch.zeros((5, 20, 24), dtype=torch.uint8, device="cuda")
    imgs[3, 7, 9] = 2
    p = gpu_lib.lpf_build_paths(6, 5)
    gpu_lib.lpf_set_checked(p, True)
    gpu_lib.lpf_full_ensemble(imgs, p)
    assert gpu_lib.lpf_paths_status(p) == gpu_lib.LPF_EPIXEL
