"""The walks that re-deal few live masks over the lanes, on calls that take
them: windows from 128 on with four or eight words per thread and enough units
(images), windows from 120 on (batches); and volumes with a window of 128 along
an axis, in every shape of tile.  References: the
oracle for the selections of translations and sampled vectors, and for
whole tables the walk with one word per thread, which never re-deals."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

CASES = [
    ("ellipses 139x163", lambda: synth.ellipses(139, 163, 0.35, seed=2, axes=(4.0, 9.0)), 131, 128),
    ("chess 149x135 full domain", lambda: synth.chess(149, 135, 10), 134, 148),
    ("lines 321x257", lambda: np.eye(321, 257, dtype=np.uint8) | np.eye(321, 257, 60, dtype=np.uint8), 128, 60),
    ("random 97x290", lambda: synth.random_binary(97, 290, 0.1, 4), 129, 96),
    ("squares 260x140", lambda: synth.squares(260, 140, 9, 0.3, seed=1), 45, 160),
]


def _units(H, W, T, n_pieces):  # at least so many, with every piece on the side of fewer tiles
    return n_pieces * min(-(-H // 32) * -(-W // (32 * T)), -(-W // 32) * -(-H // (32 * T)))


@pytest.mark.parametrize("name,make,rx,ry", CASES, ids=[c[0] for c in CASES])
def test_image_and_selection_match_the_oracle(gpu_lib, name, make, rx, ry):
    img = make()
    H, W = img.shape
    sel = (np.random.default_rng(3).random((H, W)) < 0.02).astype(np.uint8)
    base = oracle.window_sizes(rx, ry)[2]  # (sampled starts: the canonical half is the definition)
    ref_sel = oracle.lpf_full_selected(img, rx, ry, sel)[:, base:]
    d, d_sel = torch.from_numpy(img).cuda(), torch.from_numpy(sel).cuda()
    p = gpu_lib.lpf_build_paths(rx, ry)
    gpu_lib.lpf_set_launch_shape(p, H, W, 1, 1)
    ref = gpu_lib.lpf_full(d, p).cpu().numpy()
    rng = np.random.default_rng(5)
    vecs = [(int(rng.integers(-rx, rx + 1)), int(rng.integers(0, ry + 1))) for _ in range(40)]
    at = [oracle.full_index(dx, dy, rx, ry) for dx, dy in vecs]
    np.testing.assert_array_equal(ref[:, at].T, oracle.count_list(img, vecs))
    reached = 0
    for T, BB in ((4, 1), (4, 3), (8, 1), (8, 4)):
        gpu_lib.lpf_set_launch_shape(p, H, W, T, BB)
        reached += _units(H, W, T, gpu_lib.lpf_paths_stats(p)["n_pieces"]) >= 2 * 32 * 152
        np.testing.assert_array_equal(gpu_lib.lpf_full(d, p).cpu().numpy(), ref, err_msg=f"T={T} BB={BB}")
        np.testing.assert_array_equal(gpu_lib.lpf_full_mc(d, p, d_sel).cpu().numpy()[:, base:], ref_sel)
    assert reached >= 2 and gpu_lib.lpf_paths_status(p) == 0


@pytest.mark.parametrize("T", [4, 8])
def test_batch_of_wide_and_narrow_windows(gpu_lib, T):
    # the wide windows are most of the kernel's work, so it re-deals for them alone
    imgs = [synth.ellipses(139, 163, 0.35, seed=2, axes=(4.0, 9.0)), synth.chess(60, 128, 10),
            synth.squares(260, 140, 9, 0.3, seed=1)]
    radii = [(131, 119), (30, 20), (45, 160)]
    paths = [gpu_lib.lpf_build_paths(*r) for r in radii]
    b = gpu_lib.lpf_batch_create([torch.from_numpy(i).cuda() for i in imgs], paths, words_per_thread=[T] * 3)
    for i, p, c in zip(imgs, [gpu_lib.lpf_build_paths(*r) for r in radii], gpu_lib.lpf_batch_run(b)):
        gpu_lib.lpf_set_launch_shape(p, *i.shape, 1, 1)
        assert torch.equal(c, gpu_lib.lpf_full(torch.from_numpy(i).cuda(), p))
    assert gpu_lib.lpf_batch_status(b) == 0


@pytest.mark.parametrize("D,H,W,rx,ry,rz,shape", [
    (3, 150, 20, 2, 130, 1, None),        # one word per thread
    (3, 160, 50, 2, 130, 1, None),        # two words
    (3, 150, 141, 128, 5, 1, None),       # four
    (2, 160, 229, 30, 130, 1, None),      # eight
    (3, 192, 100, 2, 130, 1, None),       # three words
    (3, 256, 70, 2, 130, 1, (8, 4)),      # two bands per tile
    (3, 256, 50, 2, 130, 1, (8, 4)),      # four bands per tile
    (131, 33, 60, 1, 1, 128, None),       # the window's long axis across the slices
])
def test_volume(gpu_lib, D, H, W, rx, ry, rz, shape):
    vol = synth.boolean_spheres(D, H, W, 7.0, D * H * W // 2000, seed=W)
    d = torch.from_numpy(vol).cuda()
    p, q = (gpu_lib.lpf_build_paths_3d(rx, ry, rz) for _ in range(2))
    if shape:
        gpu_lib.lpf_set_launch_shape(p, H, W, *shape)
    gpu_lib.lpf_set_launch_shape(q, H, W, 1, 1)
    got = gpu_lib.lpf_full_3d(d, p).cpu().numpy()
    np.testing.assert_array_equal(got, gpu_lib.lpf_full_3d(d, q).cpu().numpy())
    assert gpu_lib.lpf_paths_status(p) == 0 and gpu_lib.lpf_paths_status(q) == 0
    rng = np.random.default_rng(5)
    vecs = [tuple(int(rng.integers(-r, r + 1)) for r in (rx, ry, rz)) for _ in range(40)]
    at = [oracle.full_index3(*v, rx, ry, rz) for v in vecs]
    np.testing.assert_array_equal(got[:, at].T, [[oracle.count3(vol, *v, ph) for ph in (0, 1)] for v in vecs])
