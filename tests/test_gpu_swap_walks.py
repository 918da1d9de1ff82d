"""Swap deltas that the bit planes do not serve -- cells whose extended copy
fits in shared memory and whose planes do not, segments over 255 pixels --
against the oracle's recount, and an annealing run that starts on such a cell."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

CASES = [(6000, 33, 1, 1, 5), (6, 600, 300, 2, 4), (600, 7, 3, 255, 3)]


def _pairs(cell, k):
    pairs = synth.swap_candidates(cell, k, seed=6).astype(np.int32)
    y, x = np.argwhere((cell == 1) & (np.roll(cell, -1, 1) == 0))[0]  # neighbours: segments hold both pixels
    pairs[0] = (y * cell.shape[1] + x, y * cell.shape[1] + (x + 1) % cell.shape[1])
    pairs[1] = pairs[0][::-1]
    pairs[-1] = pairs[-1][:1].repeat(2)  # the identity
    return pairs


@pytest.mark.parametrize("copies", [1, 100], ids=["few", "many"])
@pytest.mark.parametrize("H,W,rx,ry,k", CASES)
def test_exchanges_match_a_recount(gpu_lib, H, W, rx, ry, k, copies):
    cell = synth.random_binary(H, W, 0.4, seed=W)
    cell |= np.roll(cell, 1, 1)
    pairs = _pairs(cell, k)
    ref = oracle.delta_swap(cell, rx, ry, pairs)
    p = gpu_lib.lpf_build_paths(rx, ry)
    d = torch.from_numpy(cell).cuda()
    counts = gpu_lib.lpf_full(d, p)
    target = (counts.double() / cell.size * 0.9).float()
    tp = torch.from_numpy(np.tile(pairs, (copies, 1))).cuda()
    dc, de = gpu_lib.lpf_delta_swap(d, p, tp, target=target, counts=counts, want_de=True)
    assert gpu_lib.lpf_paths_status(p) == 0
    dc, de = dc.cpu().numpy().reshape(copies, k, 2, -1), de.cpu().numpy().reshape(copies, k)
    assert all(np.array_equal(c, ref) for c in dc) and (de == de[0]).all()
    # float32: at most one rounding per term and addition of a nonzero term
    ref_de = oracle.delta_objective(target.cpu().numpy(), counts.cpu().numpy(), ref, rx, ry, H, W)
    _, n_canon, base = oracle.window_sizes(rx, ry)
    dd = target.cpu().numpy()[:, base:] - counts.cpu().numpy()[:, base:] / cell.size
    mag = np.abs(ref / cell.size * (ref / cell.size - 2 * dd[None])).sum(axis=(1, 2))
    assert (np.abs(de[0] - ref_de) <= (2 * n_canon + 8) * 2.0 ** -24 * mag + 1e-12).all()
    sel = (np.random.default_rng(2).random((H, W)) < 0.3).astype(np.uint8)
    before, base = oracle.lpf_full_selected(cell, rx, ry, sel), oracle.window_sizes(rx, ry)[2]
    dc, _ = gpu_lib.lpf_delta_swap_mc(d, p, torch.from_numpy(sel).cuda(), tp)
    for q, c in zip(pairs, dc.cpu().numpy()):
        after = cell.copy()
        after.reshape(-1)[q] = after.reshape(-1)[q[::-1]]
        np.testing.assert_array_equal(c, (oracle.lpf_full_selected(after, rx, ry, sel) - before)[:, base:])


def test_annealing_finds_its_start_temperature(gpu_lib):
    H, W, r = 6000, 33, 1
    cell = synth.random_binary(H, W, 0.4, seed=1)
    target = (oracle.lpf_full(synth.clustered_disks(64, 64, 0.4, seed=2), r, r) / 4096.0).astype(np.float32)
    p = gpu_lib.lpf_build_paths(r, r)
    d = torch.from_numpy(cell).cuda()
    counts = torch.empty((2, p.n_full), dtype=torch.int64, device="cuda")
    ann = gpu_lib.lpf_sa_create(d, p, torch.from_numpy(target).cuda(), counts, n_step=200, seed=3)
    gpu_lib.lpf_sa_run(ann, 40)
    st = gpu_lib.lpf_sa_read(ann)
    assert st["t_max"] > 0 and st["n_accept"] > 0
    np.testing.assert_array_equal(counts.cpu().numpy(), oracle.lpf_full(d.cpu().numpy(), r, r))
