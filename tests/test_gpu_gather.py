"""The walk that re-deals few live masks over the lanes (windows from 64 on)
against the oracle, in every launch shape: words per thread and tiles that do
not divide the image, media that empty out early, late and never, and a
selection of translations."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

CASES = [
    ("ellipses 90x150", lambda: synth.ellipses(90, 150, 0.35, seed=2, axes=(4.0, 9.0)), 70, 40),
    ("disks 131x67", lambda: synth.disks_fixed(131, 67, 4.0, np.random.default_rng(1).uniform(0, 131, (40, 2))), 30, 64),
    ("chess 66x100 full domain", lambda: synth.chess(66, 100, 10), 99, 65),
    ("a line 40x300", lambda: np.pad(np.ones((1, 299), np.uint8), ((20, 19), (0, 1))), 200, 5),
    ("random 65x257", lambda: synth.random_binary(65, 257, 0.1, 4), 64, 9),
]


@pytest.mark.parametrize("name,make,rx,ry", CASES, ids=[c[0] for c in CASES])
def test_every_shape_matches_the_oracle(gpu_lib, name, make, rx, ry):
    img = make()
    H, W = img.shape
    ref = oracle.lpf_full(img, rx, ry)
    sel = (np.random.default_rng(3).random((H, W)) < 0.02).astype(np.uint8)
    base = oracle.window_sizes(rx, ry)[2]  # (sampled starts: the canonical half is the definition)
    ref_sel = oracle.lpf_full_selected(img, rx, ry, sel)[:, base:]
    d, d_sel = torch.from_numpy(img).cuda(), torch.from_numpy(sel).cuda()
    p = gpu_lib.lpf_build_paths(rx, ry)
    ran = 0
    for T in (1, 2, 4, 8):
        for BB in (1, 2, 4):
            try:
                gpu_lib.lpf_set_launch_shape(p, H, W, T, BB)
            except gpu_lib.LpfError:
                continue  # not a shape of this image
            np.testing.assert_array_equal(gpu_lib.lpf_full(d, p).cpu().numpy(), ref, err_msg=f"T={T} BB={BB}")
            np.testing.assert_array_equal(gpu_lib.lpf_full_mc(d, p, d_sel).cpu().numpy()[:, base:], ref_sel)
            ran += 1
    assert ran >= 6 and gpu_lib.lpf_paths_status(p) == 0


def test_batch_of_both_kinds(gpu_lib):
    # one walk kernel takes images that re-deal and images that do not
    imgs = [synth.ellipses(100, 140, 0.35, seed=2, axes=(4.0, 9.0)), synth.chess(60, 128, 10),
            synth.squares(200, 129, 4, 0.2, seed=1)]
    radii = [(69, 49), (30, 20), (64, 99)]
    paths = [gpu_lib.lpf_build_paths(*r) for r in radii]
    for T in (1, 2, 4, 8):
        b = gpu_lib.lpf_batch_create([torch.from_numpy(i).cuda() for i in imgs], paths, words_per_thread=[T] * 3)
        for i, r, c in zip(imgs, radii, gpu_lib.lpf_batch_run(b)):
            np.testing.assert_array_equal(c.cpu().numpy(), oracle.lpf_full(i, *r))
        assert gpu_lib.lpf_batch_status(b) == 0
